"""pt_autotune on ensembles that one chain per block serves best, and what it says about the units of a launch."""
import numpy as np
import pytest

import paper_2511_13508_gb300 as pkg
from paper_2511_13508_gb300 import workload

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,N,nT", [("fp32", 18, 42), ("fp64", 130, 5)])
def test_one_chain_per_block_leaves_the_groups_alone(prec, N, nT):
    """The trials rebuild the groups of the other kernels (full energies run on them too); the choice of one chain per block
    restores those of the context, to the bit of a full energy."""
    Js = [workload.couplings(N, len(pkg.enumerate_quads(N)), 3 + i) for i in range(2)]
    p = pkg.PT([N, N], Js, workload.geometric_ladder(0.3, 1.6, nT), 2, 3, precision=prec)
    p.sweep(3)
    E = p.energy()
    assert p.autotune(4)[:2] == (0, 0)
    assert np.array_equal(p.energy(), E)


def test_units_are_the_default_where_the_launch_cuts_its_own():
    """FP32 without an explicit unit: each launch cuts its runs itself, the tuner reports the default unit (8 sweeps from
    N = 48 on), whatever was timed; an explicit unit is tuned."""
    N = 64
    Js = [workload.couplings(N, len(pkg.enumerate_quads(N)), 3)]
    p = pkg.PT([N], Js, workload.geometric_ladder(0.3, 1.6, 16), 2, 3, swap_every=16, measure_every=4, resync_every=32)
    assert {p.autotune(2)[2] for _ in range(6)} == {8}
    q = pkg.PT([N], Js, workload.geometric_ladder(0.3, 1.6, 16), 2, 3, sweeps_per_unit=2)
    assert q.autotune(2)[2] in (2, 8)
