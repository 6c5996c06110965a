"""GPU: numbers that are not finite on their way through the integrand. A NaN in a factor reaches the log of every sample
that meets it, in each precision, for one- and two-sided limits, single and batched, and never counts as probability
1; limits so large that dividing them overflows count as infinite ones; a sample of probability zero (an infinite
standardised limit) counts as zero and spoils no other."""
import math

import numpy as np
import pytest
from scipy.special import log_ndtr

pytestmark = pytest.mark.gpu

PRECISIONS = ["FP64", "FP32", "BF16_SHIFT", "FP16_SHIFT"]
N, M = 200, 100  # two tiles of two 64-variable sub-tiles


@pytest.fixture(scope="module")
def tl():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__ as ge
    ge.build()
    import paper_2003_11183_gb300 as tl
    return tl


def factor(tl, where=None, n=N, m=M):
    rng = np.random.default_rng(1)
    r = n // m
    B = [np.tril(rng.normal(0.0, 0.1, (m, m)), -1) + np.eye(m) for _ in range(r)]
    U, V = {(1, 0): rng.normal(0.0, 0.1, (m, 3))}, {(1, 0): rng.normal(0.0, 0.1, (m, 3))}
    if where == "window":        # within a block of 16 variables
        B[0][70, 69] = np.nan
    elif where == "coupling":    # across sub-tiles
        B[1][90, 3] = np.nan
    elif where == "last":        # the last variable: no later one shows it
        B[1][m - 1, m - 2] = np.nan
    elif where == "U":
        U[(1, 0)][5, 1] = np.nan
    elif where == "V":
        V[(1, 0)][5, 1] = np.nan
    return tl.tlrmvn_factor_import(tl.build_export(n, m, np.arange(r + 1) * m, np.arange(n), B, U, V))


def limits(sides):
    return np.full(N, -np.inf if sides == 1 else -1.5), np.full(N, 0.7)


@pytest.mark.parametrize("where", ["window", "coupling", "last", "U", "V"])
@pytest.mark.parametrize("sides", [1, 2])
def test_nan_in_a_factor(tl, where, sides):
    F = factor(tl, where)
    a, b = limits(sides)
    for p in PRECISIONS:
        lp, _, _, pm = tl.tlrmvn_prob(F, a, b, math.inf, getattr(tl, p), 2, 100, seed=3, per_sample=True)
        assert np.all(np.isnan(pm)) and not np.isfinite(lp), p


@pytest.mark.parametrize("precision", ["FP32", "BF16_SHIFT"])
@pytest.mark.parametrize("sides", [1, 2])
def test_nan_in_a_batched_factor(tl, precision, sides):
    a, b = limits(sides)
    plan = tl.BatchPlan([factor(tl, "coupling")], math.inf, 2, 100, seed=3, precision=getattr(tl, precision))
    lp, _ = plan.run([a], [b])
    assert not np.isfinite(lp[0])
    plan.close()


@pytest.mark.parametrize("precision", PRECISIONS)
@pytest.mark.parametrize("sides", [1, 2])
def test_zero_probability_samples(tl, precision, sides):
    # x2 = x1 and x3 = x1 / 5 + x2 / 2 + z3: with x1 below 0.5 and x2 below 0.2 a sample has x2's factor 0 or 1
    B = [np.array([[1.0, 0.0, 0.0], [1.0, 0.0, 0.0], [0.2, 0.5, 1.0]])]
    F = tl.tlrmvn_factor_import(tl.build_export(3, 3, np.array([0, 3]), np.arange(3), B, {}, {}))
    a = np.full(3, -np.inf if sides == 1 else -9.0)
    lp, _, _, pm = tl.tlrmvn_prob(F, a, [0.5, 0.2, 30.0], math.inf, getattr(tl, precision), 2, 500, seed=3,
                                  per_sample=True)
    pm = np.ravel(pm)
    zero = np.isneginf(pm)
    # the samples below 0.2 are Phi(0.2) / Phi(0.5) = 0.84 of them
    assert abs(np.mean(~zero) - 0.84) < 0.02 and np.allclose(pm[~zero], log_ndtr(0.5), atol=1e-6)
    assert abs(lp - log_ndtr(0.2)) < 0.02


@pytest.mark.parametrize("precision", PRECISIONS)
@pytest.mark.parametrize("lo,hi", [(-np.inf, 1.79e308), (-1.79e308, 0.5), (-1.79e308, 1.79e308), (-np.inf, -1.79e308),
                                   (1.5e308, 1.79e308)])
def test_huge_limits(tl, precision, lo, hi):
    # a diagonal of 0.5: 1.79e308 / 0.5 is beyond float64
    B = [np.array([[0.5, 0.0, 0.0], [0.1, 0.5, 0.0], [0.2, 0.1, 0.9]])]
    F = tl.tlrmvn_factor_import(tl.build_export(3, 3, np.array([0, 3]), np.arange(3), B, {}, {}))
    inf = [math.copysign(math.inf, x) if abs(x) > 1e300 else x for x in (lo, hi)]
    got = [tl.tlrmvn_prob(F, [x, -np.inf, -9.0], [y, 0.3, 0.4], math.inf, getattr(tl, precision), 2, 100, seed=3)[0]
           for x, y in ([(lo, hi)] if max(inf) == -math.inf or min(inf) == math.inf else [(lo, hi), inf])]
    # the same as with infinite limits, which may not both lie at one end
    assert got[0] == got[1] if len(got) == 2 else np.isneginf(got[0])
