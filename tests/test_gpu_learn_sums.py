"""Bias gradients of the proposal network by number of temperature conditions and rows: one and several conditions per warp of
the column sums, more than they hold in registers, and rows that end inside and past their first piece of 128."""
import numpy as np
import pytest

import paper_2511_13508_gb300 as pkg
from oracle import learned as ol
from paper_2511_13508_gb300 import workload

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ncold,rows", [(1, 72), (8, 256), (9, 200), (64, 128), (65, 136)])
def test_bias_gradients(ncold, rows):
    N, S, nT = 16, 2, max(2, ncold)
    J = [workload.couplings(N, len(pkg.enumerate_quads(N)), 40 + s) for s in range(S)]
    pt = pkg.PT([N] * S, J, workload.geometric_ladder(0.5, 1.5, nT), 1, 5, precision="fp32")
    pt.learn_init(n_cold=ncold, batch=256, data_per_sample=256, seed=9)
    sh = pt.learn_shape()
    rng = np.random.default_rng(ncold)
    P = pt.learn_params()
    P[:, sh["ob3"]:sh["ob3"] + sh["Dout"]] = 0.3 * rng.standard_normal((S, sh["Dout"]))
    P[:, sh["oC1"]:sh["oW2"]] = 0.2 * rng.standard_normal((S, sh["oW2"] - sh["oC1"]))
    pt.set_learn_params(P)
    w = rng.gamma(0.5, 1.0, (S, rows, N))  # intensities squared on the constraint surface, uniform phases
    a = (N * w / w.sum(-1, keepdims=True)) ** 0.25 * np.exp(2j * np.pi * rng.random((S, rows, N)))
    a = a.astype(np.complex64).astype(np.complex128)
    cond = rng.integers(0, ncold, (S, rows)).astype(np.int32)
    _, _, g = pt.learn_eval(a, cond, grad=True)
    for s in range(S):
        want, _ = ol.nll_grad(P[s].astype(np.float64), a[s], cond[s], N, sh["H"], ncold, 8, emulate_bf16=True)
        got = g[s].astype(np.float64)
        for lo, hi in ((sh["ob1"], sh["oC1"]), (sh["oC1"], sh["oW2"]), (sh["ob2"], sh["oW3"]), (sh["ob3"], sh["ob3"] + sh["Dout"])):
            assert np.linalg.norm(got[lo:hi] - want[lo:hi]) < 3e-2 * np.linalg.norm(want[lo:hi])
        b1, C1 = got[sh["ob1"]:sh["oC1"]], got[sh["oC1"]:sh["oW2"]].reshape(ncold, -1)
        # the same FP32 values summed in other orders: rows 2^-24 sum|v| at most, sum|v| about sqrt(rows) |sum v|
        assert np.linalg.norm(b1 - C1.sum(0)) <= rows ** 1.5 * 2.0 ** -24 * np.linalg.norm(b1)
        assert not C1[np.setdiff1d(np.arange(ncold), cond[s])].any()
