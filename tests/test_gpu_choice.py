"""GPU: which sweep a block runs depends on the population and its state alone.

A block runs in the basis of the kernel's columns where no decision is expected within FP32's
rounding of its threshold, an estimate from the population's moves and mean residue.  Shards of
a population, a restored handle and a handle whose state was set choose as the one handle does that
ran through, on both sides of the line and at the block where a schedule crosses it.
"""
import numpy as np
import pytest

import paper_1609_07936_gb300 as sail
from paper_1609_07936_gb300.sharded import CudaShard, LocalComm, ShardedAnneal
from workloads import Peak, make_problem

pytestmark = pytest.mark.gpu


def _problem(n_tau=40, n_omega=200, power=1.5):
    tau = 8.0 * (np.arange(n_tau, dtype=np.float64) / (n_tau - 1)) ** power
    return make_problem("choice", tau, n_omega, 20.0, [Peak("lorentz", 2.0, 0.3, 0.6), Peak("lorentz", 5.0, 0.5, 0.4)], 1e-4, 3, 1)


def _new(P, prm):
    return sail.Sail(P.tau, P.F, P.sigma, P.omega, prm)


# blocks of 20 sweeps of 512 walkers x 200 bins (2e6 moves, a shard's a quarter of them or less), T from
# 10 chi2_0 down 14 decades: the population crosses the line, and a shard by itself would later
SCHEDULE = dict(n_walkers=512, n_sweeps=800, sweeps_per_block=20, resync_every=10, T_start=10.0, T_end=1e-13, seed=22)


@pytest.mark.parametrize("spans", [[(0, 256), (256, 256)], [(0, 100), (100, 301), (401, 111)]])
def test_shards_choose_as_the_population(spans):
    P = _problem()
    prm = sail.Params(A=P.A, B=P.B, resync_kind=sail.RESYNC_TENSOR_BF16, **SCHEDULE)
    whole = _new(P, prm)
    shards = [CudaShard(P.tau, P.F, P.sigma, P.omega, prm, o, n, 512) for o, n in spans]
    run = ShardedAnneal(shards, [spans], LocalComm(), prm.branch_fraction, prm.imprint_t)
    counts = []
    for _ in range(40):
        whole.anneal(1)
        run.block()
        counts.append(whole.span_info()["blocks"])
        assert [s.handle.span_info()["blocks"] for s in shards] == [counts[-1]] * len(shards)
    assert 1 < counts[-1] < 39                 # the schedule crosses the line
    ref = whole.state()
    for s in shards:
        sl = slice(s.offset, s.offset + s.n_walkers)
        for x, y in zip(s.handle.state()[:4], ref):
            np.testing.assert_array_equal(x, y[sl])
        s.close()
    whole.close()


def test_cold_shards_of_few_moves_follow_the_population():
    """64 walkers of 64 bins, blocks of 100 sweeps at T = 1e-12 chi2_0: 409600 moves, over the line; 16
    walkers' 102400 would lie under it."""
    P = _problem(32, 64)
    prm = sail.Params(A=P.A, B=P.B, n_walkers=64, n_sweeps=300, T_start=1e-12, T_end=1e-12, seed=3, resync_kind=sail.RESYNC_FP32)
    whole = _new(P, prm)
    spans = [(16 * k, 16) for k in range(4)]
    shards = [CudaShard(P.tau, P.F, P.sigma, P.omega, prm, o, n, 64) for o, n in spans]
    run = ShardedAnneal(shards, [spans], LocalComm(), prm.branch_fraction, prm.imprint_t)
    for _ in range(3):
        whole.anneal(1)
        run.block()
    ref = whole.state()
    assert whole.span_info()["blocks"] == 0
    for s in shards:
        assert s.handle.span_info()["blocks"] == 0
        for x, y in zip(s.handle.state()[:4], ref):
            np.testing.assert_array_equal(x, y[s.offset:s.offset + 16])
        s.close()
    whole.close()


@pytest.mark.parametrize("set_first", [False, True])
def test_a_resumed_run_chooses_as_the_uninterrupted_one(set_first):
    """Resumed before every block around the line, from a checkpoint of a run state and of one that was
    set: block by block the same sweeps, and the same bits at the end."""
    P = _problem()
    prm = sail.Params(A=P.A, B=P.B, resync_kind=sail.RESYNC_TENSOR_BF16, **SCHEDULE)
    g = _new(P, prm)
    if set_first:
        g.set_state(g.state()[0])
    for _ in range(25):
        h = _new(P, prm)
        h.restore(g.checkpoint())
        before = g.span_info()["blocks"]
        g.anneal(1)
        h.anneal(1)
        assert h.span_info()["blocks"] == g.span_info()["blocks"] - before
        for x, y in zip(g.state()[:4], h.state()[:4]):
            np.testing.assert_array_equal(x, y)
        h.close()
    assert 1 < g.span_info()["blocks"] < 24
    g.close()


def test_a_set_state_and_imprinted_walkers_are_known():
    """A warm start of more than 156250 moves a block, hot: its residue is known, and so is the
    residue after walkers were imprinted."""
    P = _problem()
    prm = sail.Params(A=P.A, B=P.B, n_walkers=512, sweeps_per_block=20, resync_every=10, branching=False, seed=5)
    g = _new(P, prm)
    g.set_state(g.state()[0])
    g.anneal(1)
    assert g.span_info()["blocks"] == 1
    g.imprint_rows([3, 4], *g.walker_rows([1, 2]), 0.1)
    h = _new(P, prm)
    h.restore(g.checkpoint())
    for s in (g, h):
        s.anneal(1)
    assert g.span_info()["blocks"] == 2 and h.span_info()["blocks"] == 1
    for x, y in zip(g.state()[:4], h.state()[:4]):
        np.testing.assert_array_equal(x, y)
    g.close()
    h.close()


@pytest.mark.parametrize("W", [1, 31, 33, 1024, 1025, 4099])
def test_the_mean_residue_is_the_blocks(W):
    """The mean over the population's chi2 that shards are told is the block statistics' to the bit, and a
    population of another size is refused."""
    P = _problem(5, 8)
    g = _new(P, sail.Params(A=P.A, B=P.B, n_walkers=W, sweeps_per_block=3, resync_every=3, branching=False, seed=5))
    stats = g.anneal(1)
    assert g.population_residue(g.chi2()) == stats[0]["chi2_mean"]
    with pytest.raises(sail.SailError):
        g.population_residue(np.ones(W + 1))
    g.close()
