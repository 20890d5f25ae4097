"""pt_autotune on ensembles that one chain per block serves best."""
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
