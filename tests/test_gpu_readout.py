"""Host readout of the state, which passes through the snapshot buffer in one piece or two."""
import numpy as np
import pytest

import paper_2511_13508_gb300 as pkg
from paper_2511_13508_gb300 import workload

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("Ns,R,nT", [([128] * 9, 4, 16), ([128, 34, 6], 16, 12), ([64], 2, 5)], ids=str)
def test_readout_in_pieces(Ns, R, nT):
    """FP32 without measurements has one snapshot (two pieces above 1 MB, the first two ensembles); with them it has four."""
    Js = [workload.couplings(N, len(pkg.enumerate_quads(N)), 40 + i) for i, N in enumerate(Ns)]
    kw = dict(precision="fp32", swap_every=4, resync_every=0)
    a, b = (pkg.PT(Ns, Js, workload.geometric_ladder(0.3, 1.6, nT), R, 5, measure_every=m, **kw) for m in (0, 1))
    for p in (a, b):
        p.sweep(8)
    assert np.array_equal(a.state()[0], b.state()[0]) and np.array_equal(a.state()[1], b.state()[1])
    assert np.array_equal(a.running_energies(), b.state()[1])
    x = a.state()[0]
    a.set_state(np.conj(x))
    assert np.array_equal(a.state()[0], np.conj(x))
