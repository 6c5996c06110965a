"""GPU: the float64 step's tables of Phi(-x) and Phi^-1 (csrc/sov64.cuh), per sample against mpmath and SciPy.

n = 1 gives Phi at a chosen limit in every sample; an infinite first limit gives the second of two variables
a limit that is an affine function of Phi^-1 of the lattice value.  Tolerances: a table value is rounded once and
its polynomial adds a few units of 2^-53, which a limit x amplifies by x (d log Phi / dx = phi / Phi <= x + 1).
"""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def tl():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__ as ge
    ge.build()
    import paper_2003_11183_gb300 as tl
    return tl


@pytest.mark.parametrize("x", [0.0, 1 / 128, 1.0 / 64, 0.9921875, 3.0899, 3.0901, 5.5, 8.3, 12.9921875, 12.9922, 13.0,
                               13.0001, 20.0, 37.0])
@pytest.mark.parametrize("sign", [1.0, -1.0])
def test_phi_table(tl, x, sign):
    import mpmath as mp
    b = sign * x
    with mp.workdps(60):  # (SciPy's log_ndtr(13) is off by 3e-14: it rounds 13 / sqrt(2))
        h = mp.erfc(mp.mpf(abs(b)) / mp.sqrt(2)) / 2
        want = float(mp.log(h) if b < 0 else mp.log1p(-h))
    F = tl.tlrmvn_factor_dense(np.array([[1.0]]), None, None, 1, 0.0, 0, 0)
    pm = tl.tlrmvn_prob(F, [-np.inf], [b], math.inf, tl.FP64, 1, 33, seed=3, per_sample=True)[3]
    assert np.all(pm == pm[0])
    assert abs(pm[0] - want) <= 1e-15 * (8 + x) * abs(want) + 1e-16 * (b <= 3.09) * (1 + x)


@pytest.mark.parametrize("a,b", [(-1.0, 2.0), (-13.5, 0.3), (0.4, 0.7), (2.0, 2.0001), (-0.7, -0.4), (6.0, 14.0),
                                 (-3.4, 3.5), (-14.0, 15.0), (12.5, 13.5), (-np.inf, 1.0), (1.0, np.inf), (14.0, 15.0)])
def test_intervals(tl, a, b):
    import mpmath as mp
    with mp.workdps(60):
        ea = mp.mpf(0) if np.isneginf(a) else mp.erfc(-mp.mpf(a) / mp.sqrt(2)) / 2
        ca = mp.mpf(1) if np.isneginf(a) else mp.erfc(mp.mpf(a) / mp.sqrt(2)) / 2
        cb = mp.mpf(0) if np.isposinf(b) else mp.erfc(mp.mpf(b) / mp.sqrt(2)) / 2
        eb = mp.mpf(1) if np.isposinf(b) else mp.erfc(-mp.mpf(b) / mp.sqrt(2)) / 2
        p = eb - ea if b <= 0 else ca - cb
        want = float(mp.log(p))
        spread = float(max(eb, mp.mpf(0)) / p) if b <= 0 else float(ca / p)  # cancellation of the two tails
    F = tl.tlrmvn_factor_dense(np.array([[1.0]]), None, None, 1, 0.0, 0, 0)
    pm = tl.tlrmvn_prob(F, [a], [b], math.inf, tl.FP64, 1, 33, seed=3, per_sample=True)[3]
    # (a limit's own rounding moves log p by phi / p times it; beyond the tables the step works in logs)
    assert np.all(np.abs(pm - want) <= 2e-15 * (1 + spread) * (1 + min(abs(a), abs(b)) ** 2))


@pytest.mark.parametrize("m", [1, 2])
def test_quantile_table(tl, m):
    # 3 x 5,461 lattice points: w from about 1e-4 to 1 - 1e-4, and both halves of every octave down to there
    from scipy.special import log_ndtr, ndtri
    from oracle import lattice
    r, b2, M, N = 0.8, 0.3, 3, 5461
    F = tl.tlrmvn_factor_dense(np.array([[1.0, r], [r, 1.0]]), None, None, m, 1e-14, 0, 0)
    shifts = np.random.default_rng(5).integers(0, 2 ** 64 - 1, size=(M, 3), dtype=np.uint64)
    pm = tl.tlrmvn_prob(F, [-np.inf] * 2, [np.inf, b2], math.inf, tl.FP64, M, N, shifts=shifts, per_sample=True)[3]
    w = lattice.qmc_points(lattice.richtmyer_generators(3), shifts, N)[:, 0]
    y = np.where(w <= 0.5, ndtri(w), -ndtri(1.0 - w))  # (1 - w is exact)
    want = log_ndtr((b2 - r * y) / math.sqrt(1.0 - r * r))
    assert np.max(np.abs(pm - want)) <= 5e-14
