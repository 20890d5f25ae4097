"""The FP32 J-sharing comb sweep (pt_comb.cu): blocks alone and clusters of 2, 4 and 8 blocks per group agree.

An ensemble of few groups of 8 chains runs each group on a cluster (the largest that keeps all groups resident, by N); a
limit on the blocks per SM keeps one block per group.  Proposals and random numbers are the same, the order of the sums
is not, so over few decisions (an FP32 one lies within rounding of its threshold once in 5e7) amplitudes and counters
agree and energies agree to rounding.
"""
import numpy as np
import pytest

import paper_2511_13508_gb300 as pkg
from paper_2511_13508_gb300 import workload

pytestmark = pytest.mark.gpu

CASES = [
    # Ns, replicas, temperatures: groups of 8 (partial ones too), clusters by N and count on 152 SMs
    ([64], 2, 9), ([66, 64], 1, 9), ([96], 1, 3), ([128], 2, 8), ([130, 128, 34], 2, 5), ([128] * 25, 1, 9), ([256], 2, 8),
    ([256] * 21, 1, 8), ([512], 1, 3),
]


@pytest.mark.parametrize("Ns,R,nT", CASES, ids=["%dx%d-%d" % (len(c[0]), max(c[0]), c[1] * c[2]) for c in CASES])
def test_clusters_agree_with_single_blocks(Ns, R, nT):
    by = {N: len(pkg.enumerate_quads(N)) for N in set(Ns)}
    Js = [workload.couplings(N, by[N], 40 + i) for i, N in enumerate(Ns)]
    temps = workload.geometric_ladder(0.3, 1.6, nT)
    kw = dict(precision="fp32", swap_every=3, measure_every=1, resync_every=0)
    runs = [pkg.PT(Ns, Js, temps, R, 23, **kw), pkg.PT(Ns, Js, temps, R, 23, chains_per_block=8, consumer_warps=7, **kw),
            pkg.PT(Ns, Js, temps, R, 23, chains_per_block=8, consumer_warps=11, blocks_per_sm=1, **kw)]
    n = 2 if max(Ns) >= 256 else 4
    for p in runs:
        p.sweep(n)
    (x, E), o = runs[-1].state(), runs[-1].observables()
    for p in runs[:-1]:
        y, F = p.state()
        q = p.observables()
        assert np.array_equal(x, y)
        # an update's energy change is a sum of up to 4 N^2 products of order 1/N: 1e-5 of N is 100 roundings
        assert np.abs(E - F).max() <= 1e-5 * max(Ns)
        assert np.array_equal(o["mc_acc"], q["mc_acc"]) and np.array_equal(o["mc_att"], q["mc_att"])
        assert np.array_equal(o["swap_acc"], q["swap_acc"]) and np.array_equal(o["qhist"], q["qhist"])


def test_cluster_run_equals_its_pieces():
    """Measurement points, swaps and launches cut a cluster's run without changing it; full energies agree."""
    Js = [workload.couplings(128, len(pkg.enumerate_quads(128)), 3)]
    temps = workload.geometric_ladder(0.3, 1.6, 8)
    kw = dict(swap_every=4, measure_every=2, resync_every=8)
    a, b = (pkg.PT([128], Js, temps, 2, 5, **kw) for _ in range(2))
    a.sweep(11)
    for n in (1, 6, 4):
        b.sweep(n)
    assert np.array_equal(a.state()[0], b.state()[0]) and np.array_equal(a.state()[1], b.state()[1])
    assert np.abs(a.energy() - a.state()[1]).max() <= 1e-5 * 128
