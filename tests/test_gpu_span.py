"""GPU: the span sweep (the FP32 moves in an orthonormal basis of the kernel's columns) takes the
decisions of the sweep over tau, at the edges of its layouts.

A block whose decisions lie far from FP32's rounding runs the span sweep; the sweep with FP64
acceptance near the threshold (fp64_accept = 1) always runs over tau, and where none of its
decisions changed it is the plain FP32 chain bit for bit.  At T = 10 chi2_0 both must end in the
same spectra: the spectra depend on the draws and decisions alone.  The cases cover the three basis
widths, 8 and 4 lanes per walker, the column table and the spectra in shared and in global
memory, sweeps that end inside a batch of draws, and partial walker groups.
"""
import numpy as np
import pytest

import paper_1609_07936_gb300 as sail
from workloads import Peak, make_problem

pytestmark = pytest.mark.gpu


def _problem(n_tau, n_omega, tau_max=8.0, floor=0.0):
    tau = tau_max * np.arange(n_tau, dtype=np.float64) / max(1, n_tau - 1)
    peaks = [Peak("lorentz", 2.0, 0.3, 0.6), Peak("lorentz", 5.0, 0.5, 0.4)]
    return make_problem("span", tau, n_omega, 20.0, peaks, 1e-4, 3, 1, noise_floor=floor)


def _run(P, W, **kw):
    prm = sail.Params(n_walkers=W, n_sweeps=20000, sweeps_per_block=3, resync_every=2, branching=False, A=P.A, B=P.B,
                      seed=11, trace=False, resync_kind=sail.RESYNC_FP32, **kw)
    g = sail.Sail(P.tau, P.F, P.sigma, P.omega, prm)
    stats = g.anneal(1)
    a, R, chi2, acc, _ = g.state()
    flips = g.info()["fp64_flips"]
    g.close()
    return a, R, chi2, acc, stats[0]["positivity_rejected"], flips


@pytest.mark.parametrize("n_tau,n_omega,W,tau_max,floor", [
    (1, 8, 1, 8.0, 0.0),          # one walker on one tau point
    (5, 3, 5, 8.0, 0.0),          # fewer bins than a batch of draws
    (32, 64, 64, 2.0, 0.0),       # 16 directions
    (33, 65, 4097, 4.0, 0.0),     # 4 lanes per walker, spectra in shared memory, odd sizes
    (200, 1000, 63, 8.0, 0.0),    # 24 directions, 8 lanes, everything in shared memory
    (200, 1001, 10001, 8.0, 0.0),   # 4 lanes, spectra in global memory, a partial group
    (512, 2043, 130, 8.0, 0.0),   # 8 lanes, spectra in global memory
    (96, 2600, 70, 8.0, 0.0),     # the column table in global memory
    (300, 501, 77, 40.0, 1e-3),   # 32 directions
])
def test_span_sweep_takes_the_decisions_of_the_sweep_over_tau(n_tau, n_omega, W, tau_max, floor):
    P = _problem(n_tau, n_omega, tau_max, floor)
    x = _run(P, W)
    y = _run(P, W, fp64_accept=1)
    assert y[-1] == 0
    for u, v in zip(x[:-1], y[:-1]):
        np.testing.assert_array_equal(np.asarray(u), np.asarray(v))
    assert x[3].sum() > 0


@pytest.mark.parametrize("n_omega,kw", [
    (1001, {}), (1003, {"hastings": True}), (1006, {"index_walk_len": 2}), (1001, {"index_walk_len": 3}),
    (1007, {"index_walk_len": 7, "walk_uniform": 0.2}), (1000, {"index_walk_len": 1}),
])
def test_a_restored_run_takes_the_decisions_of_the_sweep_over_tau(n_omega, kw):
    """After set_state the residue is not known and a block of more than 156250 moves runs over tau; a
    handle restored from that very state knows it and runs the span sweep.  Same spectra, accepted
    moves and positivity rejections, also where the sweep ends inside a batch of draws."""
    P = _problem(40, n_omega)
    prm = sail.Params(n_walkers=301, n_sweeps=20000, sweeps_per_block=3, branching=False, A=P.A, B=P.B, seed=11,
                      resync_kind=sail.RESYNC_FP32, **kw)
    runs = []
    g = sail.Sail(P.tau, P.F, P.sigma, P.omega, prm)
    g.set_state(g.state()[0])
    blob = g.checkpoint()
    h = sail.Sail(P.tau, P.F, P.sigma, P.omega, prm)
    h.restore(blob)
    for s in (g, h):
        stats = s.anneal(1)[0]
        runs.append((*s.state()[:4], stats["positivity_rejected"], stats["acceptance"]))
        s.close()
    for u, v in zip(*runs):
        np.testing.assert_array_equal(np.asarray(u), np.asarray(v))


def test_wide_ranges_keep_the_sweep_over_tau():
    """tau up to 150 with noise falling as e^{-tau} to 1e-12: the columns need 36 directions, 32 leave 1.2e-7
    of one, and the sweep over tau serves the problem."""
    tau = 150.0 * (np.arange(400, dtype=np.float64) / 399) ** 1.5
    P = make_problem("wide", tau, 400, 20.0, [Peak("lorentz", 2.0, 0.3, 1.0)], 1e-4, 3, 1, noise_floor=1e-3)
    sigma = 1e-2 * np.maximum(np.exp(-tau), 1e-12)
    out = []
    for guard in (0, 1):
        prm = sail.Params(n_walkers=40, n_sweeps=20000, sweeps_per_block=3, resync_every=2, branching=False, A=P.A, B=P.B,
                          seed=5, fp64_accept=guard)
        g = sail.Sail(P.tau, P.F_exact, sigma, P.omega, prm)
        g.anneal(1)
        out.append(g.state()[0])
        g.close()
    np.testing.assert_array_equal(out[0], out[1])


@pytest.mark.parametrize("n_tau,n_omega,W,tau_max,floor,width", [
    (1, 8, 1, 8.0, 0.0, 16), (5, 3, 5, 8.0, 0.0, 16), (32, 64, 64, 2.0, 0.0, 16), (33, 65, 4097, 4.0, 0.0, 24),
    (200, 1000, 63, 8.0, 0.0, 24), (200, 1001, 10001, 8.0, 0.0, 24), (512, 2043, 130, 8.0, 0.0, 24),
    (96, 2600, 70, 8.0, 0.0, 24), (300, 501, 77, 40.0, 1e-3, 32),
])
@pytest.mark.parametrize("guard", [0, 1])
def test_which_sweep_a_block_runs(n_tau, n_omega, W, tau_max, floor, width, guard):
    """The widths of the bases (the numerical ranks of these kernels at 2^-26, in numpy: 1, 3, 15, 18, 23,
    23, 23, 22 and 29) and, of the two sides that the comparison above takes, that one sweeps in the
    basis and the other over tau."""
    P = _problem(n_tau, n_omega, tau_max, floor)
    g = sail.Sail(P.tau, P.F, P.sigma, P.omega,
                  sail.Params(n_walkers=W, n_sweeps=20000, sweeps_per_block=3, resync_every=2, branching=False, A=P.A, B=P.B,
                              seed=11, resync_kind=sail.RESYNC_FP32, fp64_accept=guard))
    assert g.span_info()["blocks"] == 0
    g.anneal(2)
    assert g.span_info()["blocks"] == (0 if guard else 2)
    if not guard:
        assert g.span_info()["width"] == width
    g.close()


def test_wide_ranges_have_no_basis():
    """The problem of the test above whose columns need 36 directions."""
    tau = 150.0 * (np.arange(400, dtype=np.float64) / 399) ** 1.5
    P = make_problem("wide", tau, 400, 20.0, [Peak("lorentz", 2.0, 0.3, 1.0)], 1e-4, 3, 1, noise_floor=1e-3)
    sigma = 1e-2 * np.maximum(np.exp(-tau), 1e-12)
    prm = sail.Params(n_walkers=40, n_sweeps=20000, sweeps_per_block=3, resync_every=2, branching=False, A=P.A, B=P.B, seed=5)
    g = sail.Sail(P.tau, P.F_exact, sigma, P.omega, prm)
    g.anneal(1)
    assert g.span_info() == {"width": 0, "blocks": 0}
    g.close()


@pytest.mark.parametrize("kw", [{}, {"hastings": True}, {"index_walk_len": 2}, {"index_walk_len": 5}])
def test_batched_span_sweep_ends_as_the_problem_alone(kw):
    """Three widths in one batch, an odd number of walkers and sweeps that end inside a batch of draws."""
    probs = [(_problem(32, 61, 2.0), 16), (_problem(200, 503), 24), (_problem(300, 501, 40.0, 1e-3), 32)]
    prm = [sail.Params(n_walkers=61 + k, n_sweeps=20000, sweeps_per_block=3, resync_every=2, branching=False, A=P.A, B=P.B,
                       seed=80 + k, resync_kind=sail.RESYNC_FP32, **kw) for k, (P, _) in enumerate(probs)]
    batch = sail.Batch([(P.tau, P.F, P.sigma, P.omega, p) for (P, _), p in zip(probs, prm)], autotune=False)
    batch.anneal(2)
    for h, (P, width), p in zip(batch.handles, probs, prm):
        assert h.span_info() == {"width": width, "blocks": 2}
        alone = sail.Sail(P.tau, P.F, P.sigma, P.omega, p)
        alone.anneal(2)
        assert alone.span_info()["blocks"] == 2
        for x, y in zip(h.state()[:4], alone.state()[:4]):
            np.testing.assert_array_equal(x, y)
        alone.close()
    batch.close()
