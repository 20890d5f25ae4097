"""Block shapes of default FP32 ensembles."""
import numpy as np
import pytest

import paper_2511_13508_gb300 as pkg
from paper_2511_13508_gb300 import workload

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N", [8, 16, 32, 46])
def test_small_modes_take_16_chains_where_groups_of_8_outnumber_the_sms(N):
    """Below N = 48, groups of 8 that do not all fit at once: 16 chains a block, as equal bits of the energies show."""
    import torch
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    R, nT = -(-13 * sms * 8 // 10 // 40), 40  # 1.3 groups of 8 per SM
    Js = [workload.couplings(N, len(pkg.enumerate_quads(N)), 31)]
    kw = dict(swap_every=4, measure_every=0, resync_every=0)
    a, b = (pkg.PT([N], Js, workload.geometric_ladder(0.3, 1.6, nT), R, 11, **k) for k in (kw, dict(kw, chains_per_block=16, consumer_warps=7)))
    for p in (a, b):
        p.sweep(6)
    assert np.array_equal(a.state()[1], b.state()[1]) and np.array_equal(a.state()[0], b.state()[0])
