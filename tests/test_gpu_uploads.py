"""What the host hands over (couplings, tables, a checkpoint, parameters) is on the device before the context's stream reads
it: calls in close succession, with copies below and above the 64 KB that a copy may return ahead of, give the same bits."""
import numpy as np
import pytest

import paper_2511_13508_gb300 as pkg
from paper_2511_13508_gb300 import workload

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,Ns,R,nT", [("fp64", [66, 40], 2, 5), ("fp64", [16], 1, 3), ("fp32", [24], 2, 8), ("fp32", [96, 64], 4, 16)], ids=str)
def test_close_calls_repeat(prec, Ns, R, nT):
    Js = [workload.couplings(N, len(pkg.enumerate_quads(N)), 50 + i) for i, N in enumerate(Ns)]
    temps, kw = workload.geometric_ladder(0.3, 1.6, nT), dict(precision=prec, swap_every=2, measure_every=1, resync_every=4)
    first = None
    for _ in range(8):
        p = pkg.PT(Ns, Js, temps, R, 7, **kw)
        E0 = p.state()[1]
        blob = p.save()
        p.sweep(3)
        E = p.state()[1]
        p.load(blob)
        p.sweep(3)
        assert np.array_equal(p.state()[1], E)
        first = first or (E0, E)
        assert np.array_equal(E0, first[0]) and np.array_equal(E, first[1])
        p.close()
