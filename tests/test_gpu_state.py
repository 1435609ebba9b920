"""GPU: an FP32 state crosses to the device and back as FP64, converted there a piece at a time: the round trip
is numpy's rounding to FP32, whatever the pieces, and the residual rows come without their padding."""
import numpy as np
import pytest

import paper_1609_07936_gb300 as sail
from workloads import Peak, make_problem

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_tau,n_omega,W", [
    (1, 9, 1),            # less than a block
    (33, 65, 300),        # one piece, padded residual rows
    (64, 2048, 16),       # the buffer holds more than the state
    (200, 1001, 701),     # three pieces, the last one partial; rows across pieces
    (512, 64, 4099),      # residuals longer than spectra, eight pieces
])
def test_state_round_trip(n_tau, n_omega, W):
    tau = 8.0 * np.arange(n_tau, dtype=np.float64) / max(1, n_tau - 1)
    P = make_problem("state", tau, n_omega, 20.0, [Peak("lorentz", 2.0, 0.3, 1.0)], 1e-4, 3, 1)
    rng = np.random.default_rng(5)
    a = rng.uniform(0.0, 1.0, (W, n_omega)) * 10.0 ** rng.uniform(-42, 1, (W, n_omega))   # FP32 denormals and zeros too
    acc = rng.integers(0, n_omega, W).astype(np.int32)
    g = sail.Sail(P.tau, P.F, P.sigma, P.omega, sail.Params(n_walkers=W, A=P.A, B=P.B, seed=1))
    g.set_state(a, acc)
    got, R, chi2, acc2, _ = g.state()
    np.testing.assert_array_equal(got, a.astype(np.float32).astype(np.float64))
    np.testing.assert_array_equal(acc2, acc)
    rows, n = [], 1024
    for lo in range(0, W, n):
        rows.append([x.cpu().numpy() for x in g.walker_rows(np.arange(lo, min(lo + n, W)))])
    np.testing.assert_array_equal(got, np.concatenate([r[0] for r in rows]))
    np.testing.assert_array_equal(R, np.concatenate([r[1] for r in rows]))
    np.testing.assert_allclose(chi2, (R * R).sum(1), rtol=1e-5)
    g.close()
