"""GPU: a walker's chain is the same whether its spectrum stays in shared or in global memory.

A small population stages its spectra in shared memory, a large one leaves them in global memory,
where the lanes of a walker store its accepted moves and then fold its scale into the same array:
every lane's fold has to see the other lanes' stores.  A chain depends on the walker's own index
alone, so the walkers both populations share end in the same bits.  T is far below the residue
(or decisions are taken again in FP64 near the threshold), so the sweeps run over tau.
"""
import numpy as np
import pytest

import paper_1609_07936_gb300 as sail
from workloads import Peak, make_problem

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_tau,n_omega,W,kw", [
    (200, 1001, 12003, {"sweep_loop": 1}),                          # 8 lanes per walker
    (200, 1001, 12003, {"sweep_loop": 1, "fp64_accept": 1}),
    (200, 1001, 12003, {"sweep_loop": 1, "hastings": True}),
    (200, 1001, 12003, {"index_walk_len": 2}),
    (300, 1026, 4099, {}),                                          # 16 lanes, columns not prefetched
    (117, 1024, 12001, {"sweep_loop": 1, "sweep_lanes": 16}),
    (200, 1001, 12003, {"sweep_loop": 2}),                          # look-ahead
])
def test_global_spectra_leave_the_bits_of_staged_ones(n_tau, n_omega, W, kw):
    tau = 8.0 * np.arange(n_tau, dtype=np.float64) / (n_tau - 1)
    P = make_problem("global", tau, n_omega, 20.0, [Peak("lorentz", 2.0, 0.3, 0.6), Peak("lorentz", 5.0, 0.5, 0.4)], 1e-4, 5, 1)
    few, out = 160, []
    for n_walkers in (few, W):
        g = sail.Sail(P.tau, P.F, P.sigma, P.omega,
                      sail.Params(n_walkers=n_walkers, n_sweeps=4, sweeps_per_block=4, resync_every=2, branching=False,
                                  T_start=1e-7, T_end=1e-7, A=P.A, B=P.B, seed=57, resync_kind=sail.RESYNC_FP32, **kw))
        g.anneal(1)
        a, R, chi2, acc, _ = g.state()
        out.append((a[:few], R[:few], chi2[:few], acc[:few]))
        np.testing.assert_allclose(a.sum(1), P.A, rtol=2e-6)
        g.close()
    assert out[0][3].sum() > 0
    for x, y in zip(*out):
        np.testing.assert_array_equal(x, y)
