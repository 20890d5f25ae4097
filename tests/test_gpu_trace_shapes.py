"""Update-by-update parity (test_gpu_trace) of every block shape that users' runs take, by explicit shape: small ensembles of
default shape run one chain per block or on clusters instead.  The default routes stand beside them under their own names."""
import numpy as np
import pytest

import test_gpu_graph
import test_gpu_trace

pytestmark = pytest.mark.gpu

CASES = [
    # name, Ns, R, nT, precision, chains_per_block, consumer_warps
    ("n64_32x11", [64, 64], 2, 16, "fp32", 32, 11),
    ("n96_16x11", [96, 96], 2, 8, "fp32", 16, 11),
    ("n128_16x11", [128, 128], 2, 8, "fp32", 16, 11),
    ("ragged_16x11", [128, 32, 96, 48, 64, 96, 32], 2, 6, "fp32", 16, 11),
    ("n16_16x7", [16, 16], 2, 8, "fp32", 16, 7),
    ("n24_8x7", [24, 24], 2, 4, "fp32", 8, 7),
    ("n64_fp64_16x3", [64, 64], 2, 5, "fp64", 16, 3),
    ("n128_fp64_8x7", [128], 2, 4, "fp64", 8, 7),
    ("ragged_fp64_16x3", [40, 24, 64], 2, 3, "fp64", 16, 3),
    ("n64_clusters_8x7", [64, 64], 2, 8, "fp32", 0, 0),
    ("n160_clusters_8x7", [160], 2, 8, "fp32", 0, 0),
    ("n16_row", [16, 10], 2, 4, "fp32", 0, 0),
    ("n32_row", [32, 18], 2, 4, "fp32", 0, 0),
    ("n48_row", [48, 34], 2, 6, "fp32", 0, 0),
    ("n16_fp64_row", [16, 12], 2, 3, "fp64", 0, 0),
    ("n66_fp64_row", [66, 30], 1, 3, "fp64", 0, 0),
    ("n160_fp64_row", [160], 1, 2, "fp64", 0, 0),
]


@pytest.mark.parametrize("name,Ns,R,nT,prec,cpb,cw", CASES, ids=[c[0] for c in CASES])
def test_shape_matches_oracle(name, Ns, R, nT, prec, cpb, cw):
    test_gpu_trace.test_trace_matches_oracle(name, Ns, R, nT, prec, cpb, cw)


def _quads(N, z, seed):
    """z quadruplets of distinct modes per mode on average, drawn with repetition."""
    rng = np.random.default_rng(seed)
    q = np.sort(rng.integers(0, N, (N * z // 2, 4)), axis=1)
    return np.ascontiguousarray(q[(np.diff(q, axis=1) > 0).all(1)][: N * z // 4], np.int32)


@pytest.mark.parametrize("z,staged", [(200, True), (5400, False)])
def test_graph_group_kernel_matches_oracle(monkeypatch, z, staged):
    """The sweep of 8 chains per block: more than 352 records per update and too many modes for a pair table, with an update's
    records staged in shared memory or read from L2 as it goes."""
    N = 512
    deg = np.bincount(_quads(N, z, 920).ravel(), minlength=N).max()
    assert 2 * deg > 352 and (N * 68 + 4 + 2 * deg * 20 <= 219 * 1024) == staged
    monkeypatch.setattr(test_gpu_graph.workload, "sparse_comb_graph", lambda n, _, seed: _quads(n, z, seed))
    test_gpu_graph.test_graph_kernel_trace_matches_oracle("sparse_n512")
