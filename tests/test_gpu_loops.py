"""GPU: sweep_loop and sweep_lanes choose the FP32 move loop.

A loop or a number of lanes that is asked for sweeps every block over tau, also the small and hot
blocks that otherwise run in the basis of the kernel's columns; both take the oracle's decisions at
the edges of the draw batches and proposal windows (3 to 37 bins), of the tau chunks, and in
a batch, where each loop has kernels of its own.
"""
import numpy as np
import pytest

import oracle as O
import paper_1609_07936_gb300 as sail
from workloads import Peak, make_problem

pytestmark = pytest.mark.gpu

RUN = dict(n_sweeps=6, sweeps_per_block=6, resync_every=3, branching=False, T_start=0.5, T_end=0.5)


def _problem(n_omega, n_tau=40, n_walkers=64, power=1.0):
    tau = 3.0 * (np.arange(n_tau, dtype=np.float64) / (n_tau - 1)) ** power
    peaks = [Peak("lorentz", 2.0, 0.4, 0.6), Peak("gauss", 5.0, 0.8, 0.4)]
    return make_problem(f"loops_{n_omega}", tau, n_omega, 10.0, peaks, 1e-4, 3, n_walkers)


def _oracle(P, W, seed, **kw):
    an = O.Anneal(P.tau, P.F, P.sigma, P.omega, P.A, P.B, W, O.Schedule(seed=seed, **RUN, **kw))
    return an.run(trace=True)[0], an


def _params(P, W, seed, **kw):
    return sail.Params(n_walkers=W, A=P.A, B=P.B, trace=True, seed=seed, resync_kind=sail.RESYNC_FP32, **RUN, **kw)


def _takes(h, P, acc_o, an):
    """At least 90% of the walkers take the oracle's decisions and end in its spectra."""
    acc_g = h.trace()[0]
    assert acc_g.shape == acc_o.shape
    same = np.all(acc_g == acc_o, axis=0)
    assert same.mean() >= 0.9, same.mean()
    assert acc_o.sum() > 0 and (acc_o < P.n_omega).any()
    a = h.state()[0]
    np.testing.assert_allclose(a.sum(1), P.A, rtol=2e-6)
    for w in np.flatnonzero(same):
        np.testing.assert_allclose(a[w], an.a[w], rtol=0, atol=1e-4 * an.a[w].max())


LOOPS = [{}, {"sweep_loop": 1}, {"sweep_loop": 2}, {"sweep_lanes": 16}, {"sweep_lanes": 16, "sweep_loop": 2}]


@pytest.mark.parametrize("n_omega", [3, 5, 13, 17, 37])
@pytest.mark.parametrize("mode", [{}, {"hastings": True}])
@pytest.mark.parametrize("loop", LOOPS, ids=str)
def test_loops_take_the_oracle_decisions(n_omega, mode, loop):
    P = _problem(n_omega)
    acc_o, an = _oracle(P, 64, 23, **mode)
    g = sail.Sail(P.tau, P.F, P.sigma, P.omega, _params(P, 64, 23, **mode, **loop))
    g.anneal()
    assert g.span_info()["blocks"] == (0 if loop else 1)
    _takes(g, P, acc_o, an)
    g.close()


@pytest.mark.parametrize("n_tau,power,loop", [(5, 1.0, 1), (37, 1.0, 1), (230, 1.0, 1), (230, 1.0, 2), (40, 1.5, 1), (40, 1.5, 2),
                                              (300, 1.0, 1), (512, 1.0, 1), (512, 1.0, 0)])
def test_loops_at_the_edges_of_the_tau_chunks(n_tau, power, loop):
    P = _problem(37, n_tau, 32, power)
    acc_o, an = _oracle(P, 32, 41)
    g = sail.Sail(P.tau, P.F, P.sigma, P.omega, _params(P, 32, 41, sweep_loop=loop))
    assert g.info()["sweep_lanes"] == (8 if n_tau <= 256 and power == 1.0 else 16)
    g.anneal()
    assert g.span_info()["blocks"] == (0 if loop else 1)
    _takes(g, P, acc_o, an)
    g.close()


@pytest.mark.parametrize("mode,length", [({}, 0), ({"hastings": True}, 0), ({}, 3)])
@pytest.mark.parametrize("loop", [0, 1])
def test_batched_loops_take_the_oracle_decisions(mode, length, loop):
    """40 tau points (8 lanes over tau), 300 (16 lanes, 10 chunks) and 117 uneven ones (16 lanes, 4
    chunks) in one batch: over tau one kernel per lane count, in the basis one for all."""
    probs = [_problem(37), _problem(60, 300, 48), _problem(101, 117, 33, 1.5)]
    prms = [_params(P, P.n_walkers, 300 + k, sweep_loop=loop, index_walk_len=length, **mode) for k, P in enumerate(probs)]
    batch = sail.Batch([(P.tau, P.F, P.sigma, P.omega, prm) for P, prm in zip(probs, prms)], autotune=False)
    batch.anneal()
    assert [h.info()["sweep_lanes"] for h in batch.handles] == [8, 16, 16]
    for k, (h, P) in enumerate(zip(batch.handles, probs)):
        assert h.span_info()["blocks"] == (0 if loop else 1)
        extra = {"walk_len": length} if length else {}
        _takes(h, P, *_oracle(P, P.n_walkers, 300 + k, **mode, **extra))
    batch.close()


def test_paper_grid_blocks_over_tau_and_in_the_basis():
    """200 tau x 1000 bins x 512 walkers, two hot blocks with branching: one move at a time, looking
    ahead and in the basis, the runs end in the same bits."""
    from workloads import paper_scale_double_lorentz
    P = paper_scale_double_lorentz(1e-4, n_walkers=512)
    out, blocks = [], []
    for loop in (0, 1, 2):
        g = sail.Sail(P.tau, P.F, P.sigma, P.omega,
                      sail.Params(n_walkers=512, n_sweeps=20000, sweeps_per_block=20, resync_every=10, A=P.A, B=P.B, seed=13,
                                  sweep_loop=loop, resync_kind=sail.RESYNC_TENSOR_BF16))
        stats = g.anneal(2)
        out.append([*g.state()[:4], [s["positivity_rejected"] for s in stats]])
        blocks.append(g.span_info()["blocks"])
        g.close()
    assert blocks == [2, 0, 0]
    for other in out[1:]:
        for x, y in zip(out[0], other):
            np.testing.assert_array_equal(np.asarray(x), np.asarray(y))


@pytest.mark.parametrize("n_omega,kw", [
    (1001, {}), (1003, {"hastings": True}), (1006, {"index_walk_len": 2}), (1001, {"index_walk_len": 3}),
    (1007, {"index_walk_len": 7, "walk_uniform": 0.2}), (1000, {"index_walk_len": 1}),
])
def test_hot_blocks_count_and_end_as_over_tau(n_omega, kw):
    """Same spectra, accepted moves and positivity rejections in the basis and over tau, also where the
    sweep ends inside a batch of draws; the state was set, so its residue is taken from the walkers."""
    tau = 8.0 * np.arange(40, dtype=np.float64) / 39
    P = make_problem("hot", tau, n_omega, 20.0, [Peak("lorentz", 2.0, 0.3, 0.6), Peak("lorentz", 5.0, 0.5, 0.4)], 1e-4, 3, 1)
    out = []
    for loop in (0, 1):
        g = sail.Sail(P.tau, P.F, P.sigma, P.omega,
                      sail.Params(n_walkers=301, n_sweeps=20000, sweeps_per_block=3, branching=False, A=P.A, B=P.B, seed=11,
                                  resync_kind=sail.RESYNC_FP32, sweep_loop=loop, **kw))
        g.set_state(g.state()[0])
        stats = g.anneal(1)[0]
        assert g.span_info()["blocks"] == 1 - loop
        out.append((*g.state()[:4], stats["positivity_rejected"], stats["acceptance"]))
        g.close()
    for u, v in zip(*out):
        np.testing.assert_array_equal(np.asarray(u), np.asarray(v))
