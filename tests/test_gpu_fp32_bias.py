"""GPU: the float32 path's mean error. Its products run in accumulators that truncate, and a truncated sum is off in
the same direction for every sample, which an estimate, a mean over samples, does not average out. So the
leading parts' sums have to be exact, also where rows have many entries of one size and sign. Bound: the mean signed error of
the samples' logs against the float64 path stays below half a unit in the last place of a float32 of their size, 2^-24
of their mean (a single truncating accumulator: three times that and more)."""
import math

import numpy as np
import pytest

import synth

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


def bias(tl, F, n, b):
    shifts = np.random.default_rng(7).integers(0, 2 ** 63, size=(4, n + 1), dtype=np.uint64)
    got, want = (np.ravel(tl.tlrmvn_prob(F, np.full(n, -np.inf), np.full(n, b), math.inf, p, 4, 500, shifts=shifts,
                                         per_sample=True)[3]) for p in (tl.FP32, tl.FP64))
    return abs(np.mean(got - want)) / np.mean(np.abs(want))


@pytest.mark.parametrize("entry,diag,b", [(0.05, 0.5, -1.0), (0.05, 0.5, -5.0), (0.02, 0.3, -1.0), (0.2, 1.0, 0.0)])
def test_equal_entries(tl, entry, diag, b):
    n = 512
    B = np.tril(np.full((n, n), entry), -1) + diag * np.eye(n)
    F = tl.tlrmvn_factor_import(tl.build_export(n, n, np.array([0, n]), np.arange(n), [B], {}, {}))
    assert bias(tl, F, n, b) < 2.0 ** -24


def test_positive_entries_and_projections(tl):
    n, m, r = 2048, 256, 8
    rng = np.random.default_rng(3)
    B = [np.tril(np.abs(rng.normal(0.0, 0.03, (m, m))), -1) + 0.4 * np.eye(m) for _ in range(r)]
    U = {(i, j): np.abs(rng.normal(0.0, 0.1, (m, 4))) for i in range(r) for j in range(i)}
    V = {(i, j): np.abs(rng.normal(0.0, 0.02, (m, 4))) for i in range(r) for j in range(i)}
    F = tl.tlrmvn_factor_import(tl.build_export(n, m, np.arange(r + 1) * m, np.arange(n), B, U, V))
    assert bias(tl, F, n, -3.0) < 2.0 ** -24


@pytest.mark.parametrize("b", [-0.5, 1.0])
def test_spatial_factor(tl, b):
    w = synth.small_workload(0, 256, 61, ragged_n=2000)
    F = tl.tlrmvn_factor_kernel(w.xy, w.kernel, w.params, w.nugget, w.a, w.b, 256, 1e-5, 0, 0)
    assert bias(tl, F, 2000, b) < 2.0 ** -24
