"""The FP32 sweep kernels of explicit graphs at the edges of their ranges: few records per update (one chain per block of
two warps; up to 64 records copied ahead, more loaded as they go), pair tables of 8 and of 4 chains per block, one and
two list buffers, partial groups, ragged batches, empty lists.  Against the FP64 quadruplet-list path with the same seed:
the random numbers are the same, so over few decisions (an FP32 one lies within rounding of its threshold once in 1e7)
the chains make the same moves; amplitudes carry FP32 rounding (1e-7 per move), energies that of their sums."""
import numpy as np
import pytest

import paper_2511_13508_gb300 as pkg
from paper_2511_13508_gb300 import workload

pytestmark = pytest.mark.gpu


def random_graphs(Ns):
    g = [pkg.fmc_graph(workload.random_frequencies(N, 300 + i)) for i, N in enumerate(Ns)]
    return g, [workload.couplings(N, len(x), 60 + i) for i, (N, x) in enumerate(zip(Ns, g))]


def sparse_graphs(Ns, z):
    g = [workload.sparse_comb_graph(N, z, 500 + i) for i, N in enumerate(Ns)]
    return g, [workload.couplings(N, len(x), 70 + i) * N for i, (N, x) in enumerate(zip(Ns, g))]


CASES = [
    ("random", [4, 6], 0, 1, 3), ("random", [12, 16], 0, 2, 5), ("random", [18], 0, 2, 4), ("random", [32, 20, 26], 0, 2, 3),
    ("random", [64, 34], 0, 1, 9), ("random", [72], 0, 1, 4), ("random", [80], 0, 1, 7), ("random", [96, 64], 0, 1, 5),
    ("sparse", [64, 40], 4, 2, 5), ("sparse", [256], 16, 1, 3), ("sparse", [128], 40, 2, 2), ("sparse", [128], 70, 1, 3),
    ("sparse", [256], 100, 1, 3), ("sparse", [96], 110, 1, 3), ("sparse", [256], 160, 1, 3), ("random", [128], 0, 1, 2),
]


@pytest.mark.parametrize("kind,Ns,z,R,nT", CASES, ids=["%s-%s-z%d" % (c[0], "-".join(map(str, c[1])), c[2]) for c in CASES])
def test_fp32_graph_kernels_follow_fp64(kind, Ns, z, R, nT):
    graphs, Js = random_graphs(Ns) if kind == "random" else sparse_graphs(Ns, z)
    temps = workload.geometric_ladder(0.3, 1.6, nT)
    kw = dict(graphs=graphs, swap_every=0, measure_every=2, resync_every=0)
    a = pkg.PT(Ns, Js, temps, R, 29, precision="fp32", **kw)
    b = pkg.PT(Ns, Js, temps, R, 29, precision="fp64_plain", **kw)
    for p in (a, b):
        p.sweep(3)
        p.sweep(1)
    (x, E), (y, F) = a.state(), b.state()
    assert np.abs(x - y).max() <= 1e-5 * max(1.0, np.abs(y).max())
    assert np.abs(E - F).max() <= 1e-5 * max(max(Ns), np.abs(F).max())
    o, q = a.observables(), b.observables()
    assert np.array_equal(o["mc_acc"], q["mc_acc"]) and np.array_equal(o["mc_att"], q["mc_att"])
    assert np.allclose(o["stat"], q["stat"], rtol=1e-4, atol=1e-4)


@pytest.mark.parametrize("kind", ["random", "sparse"])
def test_runs_cut_into_launches_agree(kind):
    graphs, Js = random_graphs([32]) if kind == "random" else sparse_graphs([128], 8)
    N = len(Js) and (32 if kind == "random" else 128)
    temps = workload.geometric_ladder(0.3, 1.6, 5)
    a, b = (pkg.PT([N], Js, temps, 2, 5, precision="fp32", graphs=graphs) for _ in range(2))
    a.sweep(40)
    for n in (1, 7, 32):
        b.sweep(n)
    assert np.array_equal(a.state()[0], b.state()[0]) and np.array_equal(a.state()[1], b.state()[1])


def test_graph_without_quadruplets():
    """No interaction: every proposal is accepted at dH = 0."""
    temps = workload.geometric_ladder(0.3, 1.6, 3)
    p = pkg.PT([8], [np.zeros(0)], temps, 1, 5, precision="fp32", graphs=[np.zeros((0, 4), np.int32)])
    p.sweep(4)
    o = p.observables()
    assert np.array_equal(o["mc_acc"], o["mc_att"]) and np.all(p.state()[1] == 0.0)


@pytest.mark.parametrize("make", ["random", "sparse", "row", "comb"])
def test_contexts_of_other_sizes_keep_running(make):
    """A kernel's shared-memory limit serves every context that launches it: a larger context sweeps (with a new launch
    shape) after smaller ones were made."""
    def one(N):
        temps = workload.geometric_ladder(0.3, 1.6, 4)
        if make in ("random", "sparse"):
            graphs, Js = random_graphs([N]) if make == "random" else sparse_graphs([8 * N], 4)
            return pkg.PT([N if make == "random" else 8 * N], Js, temps, 1, 3, precision="fp32", graphs=graphs)
        Js = [workload.couplings(N, len(pkg.enumerate_quads(N)), 4)]
        kw = dict(precision="fp64") if make == "row" else dict(precision="fp32", chains_per_block=8)
        return pkg.PT([N], Js, temps, 1, 3, **kw)
    a, b = one(64), one(40)
    b.sweep(1)
    a.sweep(2)
    assert np.isfinite(a.state()[1]).all() and np.isfinite(b.state()[1]).all() and np.isfinite(a.energy()).all()
