"""GPU: the branching solve (multipliers, Delta, pairs) against the oracle at the edges of its
block: one to sixteen walkers a thread, partial last rows, and residues that are widely spread,
nearly equal, equal, or equal in clusters."""
import numpy as np
import pytest

import oracle as O
import paper_1609_07936_gb300 as sail
from workloads import tiny_double_lorentz

pytestmark = pytest.mark.gpu


def _chi2(kind, n, near=1e-10):
    rng = np.random.default_rng(n)
    x = rng.standard_normal(n)
    if kind == "spread":
        return 1e3 * np.exp(0.3 * x)
    if kind == "heavy":
        return np.exp(5.0 * x)
    if kind == "near":
        return 1e12 * (1.0 + near * np.abs(x))
    if kind == "equal":
        return np.full(n, 17.0)
    return np.repeat(100.0 + np.abs(x[: (n + 6) // 7]), 7)[:n]      # clusters of seven


@pytest.mark.parametrize("precision", [sail.PREC_FP64, sail.PREC_FP32])
@pytest.mark.parametrize("kind", ["spread", "heavy", "near", "equal", "clusters"])
@pytest.mark.parametrize("n", [2, 3, 33, 1024, 1025, 4097, 8193, 16384])
def test_solve_gives_the_oracle_multipliers(n, kind, precision):
    P = tiny_double_lorentz()
    g = sail.Sail(P.tau, P.F, P.sigma, P.omega,
                  sail.Params(n_walkers=2, precision=precision, n_sweeps=10, branching=False, A=P.A, B=P.B, seed=5,
                              walker_total=16384))
    for block, fraction in ((0, 0.25), (3, 0.6)):
        # an FP32 population's mean is summed in another order than the oracle's: its residues are kept
        # far enough apart that the sum's rounding cannot reorder break points
        c = _chi2(kind, n, 1e-10 if precision == sail.PREC_FP64 else 1e-4)
        m, delta, zero, donor = g.branch_solve(c, block, fraction)
        m_o, delta_o = O.branch_multipliers(c, O.xi_for_block(5, block, n), fraction)[:2]
        np.testing.assert_array_equal(m, m_o)
        assert delta == delta_o
        np.testing.assert_array_equal(zero, np.flatnonzero(m == 0)[: zero.size])
        np.testing.assert_array_equal(donor, np.repeat(np.arange(n), np.maximum(m - 1, 0))[: zero.size])
        assert zero.size == (m == 0).sum()
    g.close()


@pytest.mark.parametrize("precision", [sail.PREC_FP64, sail.PREC_FP32])
@pytest.mark.parametrize("n", [2, 33, 64, 65, 1024, 1025, 4097, 8193, 16384])
def test_solve_of_a_population_with_close_residues(n, precision):
    """Residues within 1e-10 of each other and less: z = (chi2 - min) / (mean - min) hangs on the mean's last
    bits, so the solve is the oracle's only if its sum is rounded like the oracle's, one walker after
    the other; also where most additions are ties (residues on a grid of 2^-13 near 2^40), and where
    the sum passes many binades, ends in the first, or holds zeros."""
    P = tiny_double_lorentz()
    g = sail.Sail(P.tau, P.F, P.sigma, P.omega,
                  sail.Params(n_walkers=2, precision=precision, n_sweeps=10, branching=False, A=P.A, B=P.B, seed=5,
                              walker_total=16384))
    rng = np.random.default_rng(n)
    ramp = np.sort(np.exp(12.0 * rng.standard_normal(n)))
    huge = np.zeros(n)
    huge[0] = 1e6
    cases = [_chi2("near", n, 1e-10), _chi2("near", n, 1e-12), _chi2("near", n, 1e-14),
             2.0**40 + rng.integers(0, 200, n) / 8192.0, ramp, ramp[::-1], huge, np.where(rng.random(n) < 0.5, 0.0, 3.0)]
    for c in cases:
        for block in range(3):
            m, delta, _, _ = g.branch_solve(c, block, 0.25)
            m_o, delta_o = O.branch_multipliers(c, O.xi_for_block(5, block, n), 0.25)[:2]
            assert delta == delta_o
            np.testing.assert_array_equal(m, m_o)
    g.close()


@pytest.mark.parametrize("precision", [sail.PREC_FP64, sail.PREC_FP32])
@pytest.mark.parametrize("scale", [1e-300, 1e-60, 1e-48, 1e-44, 1e-41, 1e-38, 1e30, 1e35, 1e37, 1e38, 1e39, 1e41, 1e44, 1e47, 1e60, 1e290, 1e296])
def test_solve_at_any_scale_of_the_residues(scale, precision):
    """The multipliers depend on the residues' ratios alone: residues whose differences, mean or its inverse
    leave FP32's range, at either end, give the oracle's; also where one walker lies far above all the
    others, whose z is then small and Delta large."""
    P = tiny_double_lorentz()
    g = sail.Sail(P.tau, P.F, P.sigma, P.omega,
                  sail.Params(n_walkers=2, precision=precision, n_sweeps=10, branching=False, A=P.A, B=P.B, seed=5,
                              walker_total=16384))
    for n in (33, 1025, 4097):
        x = np.random.default_rng(n).standard_normal(n)
        far = np.exp(0.3 * x)
        far[n // 2] = 1e8
        for c in (np.exp(0.3 * x), np.exp(5.0 * np.minimum(x, 2.0)), 1.0 + 1e-3 * np.abs(x), far):
            for block in range(2):
                m, delta, _, _ = g.branch_solve(scale * c, block, 0.25)
                m_o, delta_o = O.branch_multipliers(scale * c, O.xi_for_block(5, block, n), 0.25)[:2]
                assert delta == delta_o
                np.testing.assert_array_equal(m, m_o)
    g.close()
