"""Runs of updates of the FP32 comb sweep.  With a few more groups than the device holds at once, a launch cuts every group's
updates into runs that end in the middle of a sweep and are resumed on other SMs, with measurements in between; an explicit
unit as long as the segment keeps one run per group.  Same block shape, so every bit has to agree."""
import numpy as np
import pytest

import paper_2511_13508_gb300 as pkg
from paper_2511_13508_gb300 import workload

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("Ns,G,w", [([64], 8, 11), ([48], 8, 7), ([64, 4, 48, 16], 8, 11), ([128, 6, 96], 8, 7), ([64, 18], 16, 11)],
                         ids=str)
def test_runs_cut_in_a_sweep_change_nothing(Ns, G, w):
    import torch
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    R, nT, seg = 4, 16, 7
    S = -(-(sms * 21 // 20) * G // (R * nT))  # about 5% more groups than SMs
    Ns = [Ns[i % len(Ns)] for i in range(S)]
    nq = {N: len(pkg.enumerate_quads(N)) for N in set(Ns)}
    Js = [workload.couplings(N, nq[N], 40 + i) for i, N in enumerate(Ns)]
    kw = dict(swap_every=seg, measure_every=1, resync_every=0, chains_per_block=G, consumer_warps=w)
    temps = workload.geometric_ladder(0.3, 1.6, nT)
    a, b = pkg.PT(Ns, Js, temps, R, 9, **kw), pkg.PT(Ns, Js, temps, R, 9, sweeps_per_unit=seg, **kw)
    for p in (a, b):
        p.sweep(2 * seg)  # two launches
        p.sweep(3)
    assert np.array_equal(a.state()[0], b.state()[0]) and np.array_equal(a.state()[1], b.state()[1])
    o, q = a.observables(), b.observables()
    for k in o:
        assert np.array_equal(o[k], q[k]), k
    assert np.all(o["mc_att"] == np.array([R * (2 * seg + 3) * (N // 2) for N in Ns])[:, None])
