"""GPU: variables of infinite variance (a flat prior) in a covariance: an infinite pivot, a column of zeros below it and
the rest of the factor as without it, at places around the 64-wide Cholesky panels and their 16-wide blocks. The
block after the one with the pivot is factored like any other. Tolerance: 1e-12, the float64 factor's rounding."""
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


def cholesky(S):
    A, n = S.copy(), len(S)
    L = np.zeros_like(S)
    for k in range(n):
        L[k, k] = math.sqrt(A[k, k])
        L[k + 1:, k] = A[k + 1:, k] / L[k, k]
        A[k + 1:, k + 1:] -= np.outer(L[k + 1:, k], L[k + 1:, k])
    return L


@pytest.mark.parametrize("n,flat", [(3, [1]), (64, [0]), (130, [15, 16, 63]), (130, [64, 129]), (100, [5, 70])])
def test_infinite_variance(tl, n, flat):
    x = np.random.default_rng(n).random((n, 2))
    S = np.exp(-np.linalg.norm(x[:, None] - x[None], axis=2) / 0.3) + 1e-3 * np.eye(n)
    S[flat, flat] = np.inf
    F = tl.tlrmvn_factor_dense(S, None, None, n, 1e-12, 0, 0)
    B = np.tril(tl.parse_export(tl.tlrmvn_factor_export(F)).B[0])
    want = cholesky(S)
    big = np.isinf(want)
    assert np.array_equal(np.isinf(B), big) and big.sum() == len(flat)
    assert np.max(np.abs(B[~big] - want[~big])) < 1e-12
    for p in (tl.FP64, tl.FP32):
        assert np.isfinite(tl.tlrmvn_prob(F, np.full(n, -np.inf), np.full(n, 0.5), math.inf, p, 2, 50)[0])
