"""The one-chain-per-block sweep kernel (pt_row.cu): FP64 contexts of default shape up to N = 160, FP32 ones of small N.

Against the J-sharing block kernel (an explicit chains_per_block) with the same seed: the proposals are the same, and
FP64 sums differ by rounding only, so states and counters agree.  Sizes at the edges of the variants (rows of at most
8 and 16 pairs, longer rows, a row warp more), the smallest and the largest N, and ragged batches, through
measurements, swaps and resyncs.
"""
import numpy as np
import pytest

import paper_2511_13508_gb300 as pkg
from paper_2511_13508_gb300 import workload

pytestmark = pytest.mark.gpu

CASES = [
    ("fp64", [4], 8), ("fp64", [16, 14], 16), ("fp64", [18, 4, 30], 8), ("fp64", [32], 16), ("fp64", [34, 6, 62], 8),
    ("fp64", [64], 16), ("fp64", [66, 16], 8), ("fp64", [128], 8), ("fp64", [160, 8], 8),
    ("fp32", [4], 8), ("fp32", [16, 10], 16), ("fp32", [18, 32, 6], 32), ("fp32", [32], 8),
]


@pytest.mark.parametrize("prec,Ns,G", CASES, ids=["%s-%s" % (c[0], "-".join(map(str, c[1]))) for c in CASES])
def test_row_kernel_follows_the_block_kernel(prec, Ns, G):
    Js = [workload.couplings(N, len(pkg.enumerate_quads(N)), 900 + i) for i, N in enumerate(Ns)]
    temps = workload.geometric_ladder(0.3, 1.6, 5)
    kw = dict(precision=prec, swap_every=4, measure_every=2, resync_every=8)
    a = pkg.PT(Ns, Js, temps, 2, 17, **kw)
    b = pkg.PT(Ns, Js, temps, 2, 17, chains_per_block=G, **kw)
    n = 3 if max(Ns) > 100 else 9  # few decisions: an FP32 one lies within rounding of its threshold once in 5e7
    for p in (a, b):
        p.sweep(n)
        p.sweep(2)
    (x, E), (y, F) = a.state(), b.state()
    # amplitudes never pass through a sum; energies are sums of up to 4|Q|/N terms per update, relative rounding
    # 1e-16 / 1e-7 each against |E| of order N
    tol = 1e-12 if prec == "fp64" else 1e-5
    assert np.abs(x - y).max() <= (1e-13 if prec == "fp64" else 1e-6)
    assert np.abs(E - F).max() <= tol * max(Ns)
    o, q = a.observables(), b.observables()
    for k in o:
        if o[k].dtype == np.uint64:
            assert np.array_equal(o[k], q[k]), k
        else:
            assert np.allclose(o[k], q[k], rtol=10 * tol, atol=10 * tol), k


def test_row_kernel_resumes_bit_identically():
    """The pair products are rebuilt from the amplitudes at each launch: cutting a run into launches changes nothing."""
    Js = [workload.couplings(24, len(pkg.enumerate_quads(24)), 3)]
    temps = workload.geometric_ladder(0.3, 1.6, 6)
    for prec in ("fp64", "fp32"):
        a = pkg.PT([24], Js, temps, 2, 5, precision=prec)
        b = pkg.PT([24], Js, temps, 2, 5, precision=prec)
        a.sweep(40)
        for n in (1, 7, 32):
            b.sweep(n)
        assert np.array_equal(a.state()[0], b.state()[0]) and np.array_equal(a.state()[1], b.state()[1])
