"""One-chain-per-block sweeps (pt_row.cu) at the limits of their range: the longer FP32 rows (N = 34 ... 48), limits on the blocks per
SM, which keep an ensemble on the J-sharing blocks, the smallest N, and temperatures whose inverse is infinite."""
import numpy as np
import pytest

import paper_2511_13508_gb300 as pkg
import test_gpu_row
from paper_2511_13508_gb300 import workload

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("Ns,G", [([34, 6], 8), ([48, 34, 16], 8), ([40], 16)], ids=str)
def test_long_fp32_rows_follow_the_block_kernel(Ns, G):
    test_gpu_row.test_row_kernel_follows_the_block_kernel("fp32", Ns, G)


@pytest.mark.parametrize("prec", ["fp64", "fp32", "fp64_plain"])
def test_zero_energy_change_is_accepted_at_infinite_beta(prec):
    """Without couplings dH = 0, which is accepted at every temperature, 1 / T overflowing or not."""
    p = pkg.PT([8], [np.zeros(len(pkg.enumerate_quads(8)))], [1e-310, 0.5, 1.0], 2, 3, precision=prec, swap_every=0,
               measure_every=0, resync_every=0)
    p.sweep(5)
    o = p.observables()
    assert np.all(o["mc_att"] == 2 * 5 * 4) and np.array_equal(o["mc_acc"], o["mc_att"])


@pytest.mark.parametrize("prec,N,G,w", [("fp64", 64, 16, 3), ("fp64", 128, 8, 7), ("fp32", 16, 16, 7)])
def test_a_limit_on_the_blocks_keeps_the_block_kernel(prec, N, G, w):
    """The kernels' energies differ by rounding, so equal bits mean the same kernel."""
    Js = [workload.couplings(N, len(pkg.enumerate_quads(N)), 31)]
    kw = dict(precision=prec, swap_every=4, measure_every=0, resync_every=0)
    temps = workload.geometric_ladder(0.3, 1.6, 9)
    runs = [pkg.PT([N], Js, temps, 2, 11, blocks_per_sm=1, **kw), pkg.PT([N], Js, temps, 2, 11, **kw),
            pkg.PT([N], Js, temps, 2, 11, chains_per_block=G, consumer_warps=w, blocks_per_sm=1, **kw)]
    for p in runs:
        p.sweep(6)
    E = [p.state()[1] for p in runs]
    assert np.array_equal(E[0], E[2]) and not np.array_equal(E[1], E[2])


def test_small_fp64_launches():
    """N = 4: with more than 16 chains per SM the J-sharing blocks sweep, with fewer a block per chain does."""
    import torch
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    Js = [workload.couplings(4, len(pkg.enumerate_quads(4)), 31)]
    kw = dict(precision="fp64", swap_every=4, measure_every=0, resync_every=0)
    for R, row in ((sms // 2, True), (2 * sms + 1, False)):  # 8 temperatures
        temps = workload.geometric_ladder(0.3, 1.6, 8)
        a, b = pkg.PT([4], Js, temps, R, 11, **kw), pkg.PT([4], Js, temps, R, 11, chains_per_block=16, **kw)
        for p in (a, b):
            p.sweep(30)
        (x, E), (y, F) = a.state(), b.state()
        assert np.abs(x - y).max() <= 1e-13 and np.abs(E - F).max() <= 1e-11
        assert np.array_equal(E, F) != row
