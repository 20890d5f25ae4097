"""Swap passes against the oracle: many ladders of a few temperatures, several of which share a warp (from 2001 ladders on), in
numbers that fill no block; a warp per ladder otherwise, up to and past its tile of 256."""
import numpy as np
import pytest

import oracle
import paper_2511_13508_gb300 as pkg
from paper_2511_13508_gb300 import workload

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("S,R,nT", [(1, 1, 2), (3, 37, 2), (1, 2001, 2), (3, 700, 2), (1, 130, 3), (1, 2003, 3), (3, 701, 4), (1, 2000, 4),
                                    (1, 2001, 5), (2, 3, 17), (1, 5, 32), (1, 3, 33), (1, 2, 257), (1, 3, 258), (2, 1, 300), (1, 1, 514)])
def test_swap_passes_match_the_oracle(S, R, nT):
    Ns = [4] * S
    Js = [3.0 * workload.couplings(4, len(oracle.enumerate_quads(4)), 7 + s) for s in range(S)]
    temps = workload.geometric_ladder(0.05, 1.6, nT)
    kw = dict(swap_every=1, measure_every=2, resync_every=0)
    ref, pt = oracle.OraclePT(Ns, Js, temps, R, 19, **kw), pkg.PT(Ns, Js, temps, R, 19, precision="fp64", **kw)
    for p in (ref, pt):
        p.sweep(6)
        p.swap()
    # FP64 trajectories follow the oracle to rounding (a decision on its threshold has odds of 1e-12 each)
    (x, E), (y, F) = ref.state(), pt.state()
    assert np.abs(x - y).max() <= 1e-9 and np.abs(E - F).max() <= 1e-9
    o, q = ref.observables(), pt.observables()
    for k in ("swap_acc", "swap_att", "mc_acc", "mc_att", "qhist"):
        assert np.array_equal(np.asarray(o[k]).ravel(), np.asarray(q[k]).ravel()), k
    assert q["swap_acc"].sum() > 0
