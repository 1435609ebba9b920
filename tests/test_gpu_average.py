"""GPU: the stochastic average of an FP32 population (partial sums over parts of the walkers and
bins) against numpy sums over the same walkers, at the edges of its parts: one walker, fewer
walkers than parts, partial bin tiles, and a cut that leaves some walkers out."""
import numpy as np
import pytest

import oracle as O
import paper_1609_07936_gb300 as sail
from workloads import Peak, make_problem

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_tau,n_omega,W,factor", [(3, 9, 1, 1.5), (33, 128, 7, 1.02), (40, 129, 65, 1.05),
                                                    (200, 300, 1025, 1.02), (64, 17, 2049, 1e9)])
def test_average_is_the_sum_over_the_selected_walkers(n_tau, n_omega, W, factor):
    tau = 3.0 * np.arange(n_tau, dtype=np.float64) / (n_tau - 1)
    P = make_problem("average", tau, n_omega, 10.0, [Peak("lorentz", 2.0, 0.4, 0.6), Peak("gauss", 5.0, 0.8, 0.4)], 1e-4, 3, W)
    g = sail.Sail(P.tau, P.F, P.sigma, P.omega,
                  sail.Params(n_walkers=W, n_sweeps=400, sweeps_per_block=20, resync_every=10, branching=False, A=P.A, B=P.B,
                              seed=3, avg_chi2_factor=factor))
    g.anneal(1)
    a, _, chi2, _, _ = g.state()
    mean, err, used, c2 = g.average()
    g.close()
    sel = a[chi2 <= factor * chi2.min()]
    assert used == len(sel)
    assert W < 7 or factor > 2 or 0 < used < W
    # FP64 sums of FP32 values: 2049 additions of relative rounding 1.1e-16, in any order
    np.testing.assert_allclose(mean, sel.mean(0), rtol=1e-12, atol=1e-13 * a.max())
    want = sel.std(0, ddof=1) / np.sqrt(used) if used > 1 else np.zeros(n_omega)
    # the squares' sum: (a - mean) to 1e-13 of the largest value, over a spread
    np.testing.assert_allclose(err, want, rtol=1e-10, atol=1e-12 * a.max())
    K, Fh, _ = O.tables(P.tau, P.F, P.sigma, P.omega)
    _, want_c2 = O.residual(K, Fh, mean)
    np.testing.assert_allclose(c2, want_c2, rtol=1e-12)
