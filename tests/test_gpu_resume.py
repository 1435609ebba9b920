"""GPU: checkpoint and resume in the middle of a schedule.

The random numbers are counter-based (Philox keyed by walker, sweep and move), so a run's
future depends only on its state: the spectra, residuals and chi2 as stored, the acceptance of
the last sweep, the schedule's position and, for the paper's protocol, the temperatures set so
far and the adaptive-branching and freeze-out state.  A handle that stops after some blocks,
writes a checkpoint, and a new handle that loads it and runs the remaining blocks end bit for
bit like one uninterrupted run: FP64 and FP32 paths, branching, the self-cooling schedule with
adaptive branching and smoothing, and the trace.
"""
import numpy as np
import pytest

import paper_1609_07936_gb300 as sail
from workloads import paper_scale_double_lorentz, tiny_double_lorentz

pytestmark = pytest.mark.gpu


def _params(P, precision, protocol, W):
    kw = dict(n_walkers=W, precision=precision, n_sweeps=700, sweeps_per_block=100, resync_every=50,
              branching=True, T_start=1.0, T_end=1e-6, A=P.A, B=P.B, seed=5, trace=True,
              resync_kind=sail.RESYNC_TENSOR_BF16)
    if protocol:
        kw.update(schedule_kind=sail.SCHEDULE_SELF_COOLING, adaptive_branching=True, smooth_s=1e-2)
    return sail.Params(**kw)


def _final(g):
    a, R, chi2, acc, h = g.state()
    acc_tr, m_tr, d_tr = g.trace()
    mean, err, used, c2 = g.average()
    return a, R, chi2, acc, h, acc_tr, m_tr, d_tr, mean, c2


@pytest.mark.parametrize("precision,protocol,W", [(sail.PREC_FP64, False, 32), (sail.PREC_FP64, True, 32),
                                                  (sail.PREC_FP32, False, 256), (sail.PREC_FP32, True, 256)])
def test_resumed_run_equals_the_uninterrupted_one(precision, protocol, W):
    P = tiny_double_lorentz() if precision == sail.PREC_FP64 else paper_scale_double_lorentz(1e-4, n_walkers=W)
    prm = _params(P, precision, protocol, W)
    whole = sail.Sail(P.tau, P.F, P.sigma, P.omega, prm)
    whole.anneal()
    ref = _final(whole)
    whole.close()

    first = sail.Sail(P.tau, P.F, P.sigma, P.omega, prm)
    first.anneal(3)
    blob = first.checkpoint()
    first.close()
    second = sail.Sail(P.tau, P.F, P.sigma, P.omega, prm)
    second.restore(blob)
    assert second.info()["sweeps_done"] == 300
    stats = second.anneal()
    assert len(stats) == 4 and stats[0]["block"] == 3
    out = _final(second)
    second.close()
    for x, y in zip(ref, out):
        np.testing.assert_array_equal(np.asarray(x), np.asarray(y))


def test_restore_refuses_another_problem():
    P = tiny_double_lorentz()
    prm = _params(P, sail.PREC_FP32, False, 16)
    g = sail.Sail(P.tau, P.F, P.sigma, P.omega, prm)
    g.anneal(1)
    blob = g.checkpoint()
    prm2 = _params(P, sail.PREC_FP32, False, 16)
    prm2.seed = 6
    h = sail.Sail(P.tau, P.F, P.sigma, P.omega, prm2)
    with pytest.raises(sail.SailError):
        h.restore(blob)
    with pytest.raises(sail.SailError):
        g.restore(blob[:100])
    g.close()
    h.close()


def test_resumed_run_keeps_the_automatic_move_loop():
    """The automatic loop follows the last block's rejections, which a resumed run knows: 16 walkers a SM
    on the to-target schedule (about 25% rejections) move one at a time after the first block, as
    the uninterrupted run does.  A buffer without that share (of an earlier library) is still taken."""
    import torch
    W = 16 * torch.cuda.get_device_properties(0).multi_processor_count
    P = paper_scale_double_lorentz(1e-4, n_walkers=W)
    prm = sail.Params(n_walkers=W, n_sweeps=20000, sweeps_per_block=20, resync_every=10, T_start_abs=1e6, T_end_abs=0.03,
                      move_scale=0.1 / P.n_omega, A=P.A, B=P.B, seed=8, resync_kind=sail.RESYNC_TENSOR_BF16)
    g = sail.Sail(P.tau, P.F, P.sigma, P.omega, prm)
    stats = g.anneal(2)
    assert stats[-1]["positivity_rejected"] < 0.30 and g.info()["sweep_ahead"] == 0
    blob = g.checkpoint()
    h = sail.Sail(P.tau, P.F, P.sigma, P.omega, prm)
    assert h.info()["sweep_ahead"] == 1
    h.restore(blob)
    assert h.info()["sweep_ahead"] == 0
    for s in (g, h):
        s.anneal(2)
    for x, y in zip(g.state()[:4], h.state()[:4]):
        np.testing.assert_array_equal(x, y)
    h.restore(blob[:-8])
    assert h.info()["sweeps_done"] == 40 and h.info()["sweep_ahead"] == 1
    with pytest.raises(sail.SailError):
        h.restore(blob[:-9])
    g.close()
    h.close()
