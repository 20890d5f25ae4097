"""Host readout of the state, which passes through the snapshot buffer in one piece or two, and of full energies of FP32 chains on
either kernel (tiles, or items where many groups have few modes)."""
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


@pytest.mark.parametrize("N,S,R,nT", [(4, 3, 100, 8), (16, 1, 300, 9), (30, 5, 64, 8), (32, 5, 64, 8), (16, 2, 3, 5)])
def test_full_energies_follow_fp64(N, S, R, nT):
    Js = [workload.couplings(N, len(pkg.enumerate_quads(N)), 80 + i) for i in range(S)]
    temps = workload.geometric_ladder(0.3, 1.6, nT)
    kw = dict(swap_every=2, measure_every=0, resync_every=0)
    a, b = pkg.PT([N] * S, Js, temps, R, 5, precision="fp32", **kw), pkg.PT([N] * S, Js, temps, R, 5, precision="fp64", **kw)
    a.sweep(5)
    b.set_state(a.state()[0])
    # products and sums of 8 in FP32 (6e-8 each), of H of order N
    assert np.abs(a.energy() - b.energy()).max() <= 1e-6 * N
    a.resync()
    assert np.abs(a.running_energies() - a.energy()).max() == 0.0
