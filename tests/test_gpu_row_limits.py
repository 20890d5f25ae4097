"""One-chain-per-block sweeps (pt_row.cu) at the limits of their range: temperatures whose inverse is infinite."""
import numpy as np
import pytest

import paper_2511_13508_gb300 as pkg

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["fp64", "fp32", "fp64_plain"])
def test_zero_energy_change_is_accepted_at_infinite_beta(prec):
    """Without couplings dH = 0, which is accepted at every temperature, 1 / T overflowing or not."""
    p = pkg.PT([8], [np.zeros(len(pkg.enumerate_quads(8)))], [1e-310, 0.5, 1.0], 2, 3, precision=prec, swap_every=0,
               measure_every=0, resync_every=0)
    p.sweep(5)
    o = p.observables()
    assert np.all(o["mc_att"] == 2 * 5 * 4) and np.array_equal(o["mc_acc"], o["mc_att"])
