"""GPU: handles in different threads launch the same kernels with different shared memory.

Every handle is used by one thread and has a stream of its own; the kernels, and the largest shared
memory a launch of them may ask for, are the process's.  Runs of two problems whose kernels are
the same and whose needs differ go on side by side in two threads, and end as they do alone.
"""
import threading

import numpy as np
import pytest
import torch

import paper_1609_07936_gb300 as sail
from workloads import Peak, make_problem

pytestmark = pytest.mark.gpu


def _problem(n_omega, n_tau):
    tau = 8.0 * np.arange(n_tau, dtype=np.float64) / (n_tau - 1)
    return make_problem("threads", tau, n_omega, 20.0, [Peak("lorentz", 2.0, 0.3, 0.6), Peak("lorentz", 5.0, 0.5, 0.4)], 1e-4, 3, 1)


def _side_by_side(work):
    """Runs every function of work in a thread of its own; their results, or the first error."""
    out, errors = [None] * len(work), []

    def call(k):
        try:
            torch.cuda.set_device(0)
            out[k] = work[k]()
        except Exception as e:      # noqa: BLE001 (reported below)
            errors.append(e)

    threads = [threading.Thread(target=call, args=(k,)) for k in range(len(work))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    if errors:
        raise errors[0]
    return out


# 900 and 1000 bins hold 86 and 96 KB of the basis's columns, over tau 31 and 34 KB of factors; FP64
# stages 5600 or 6400 bins of a walker
@pytest.mark.parametrize("sizes,kw", [
    ((1000, 900), dict(n_sweeps=600)),
    ((1000, 900), dict(n_sweeps=600, sweep_loop=1)),
    ((1000, 900), dict(n_sweeps=600, shared_bins=4)),
    ((6400, 64), dict(n_sweeps=60, precision=sail.PREC_FP64)),
])
def test_sweeps_side_by_side(sizes, kw):
    def run(n_omega):
        P = _problem(n_omega, 200 if kw.get("precision") is None else 20)
        prm = sail.Params(n_walkers=8, sweeps_per_block=20, resync_every=1, A=P.A, B=P.B, seed=5, **kw)
        if n_omega == 64:           # as many launches in the time of the larger one's
            prm.n_sweeps *= 50
        with torch.cuda.stream(torch.cuda.Stream()):
            g = sail.Sail(P.tau, P.F, P.sigma, P.omega, prm)
            g.anneal()
            out = g.state()
            g.close()
        return out

    alone = [run(n) for n in sizes]
    for x, y in zip(alone, _side_by_side([lambda n=n: run(n) for n in sizes])):
        for u, v in zip(x, y):
            np.testing.assert_array_equal(u, v)
