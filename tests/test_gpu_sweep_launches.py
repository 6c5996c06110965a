"""GPU: the whole-tile sweep's launches: more tiles than one launch takes (16,384 variables; also more column ranks
than are staged at a time), more samples than the SMs hold in one pass (equal passes), and few samples, whose products
overlap the sweep.  Tolerance: the float32 path's 1e-4 relative per sample against the float64
path; passes of another size, overlapped or not, give the same bits."""
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


def _factor(tl, n, m, M, N):
    w = synth.small_workload(0, m, 500 + m, n_shifts=M, n_points=N, ragged_n=n)
    return w, tl.tlrmvn_factor_kernel(w.xy, w.kernel, w.params, w.nugget, w.a, w.b, m, w.tol, 0, 0)


def test_tiles_beyond_one_launch(tl):
    w, F = _factor(tl, 16460, 64, 2, 100)
    got = tl.tlrmvn_prob(F, w.a, w.b, math.inf, tl.FP32, 2, 100, shifts=w.shifts, per_sample=True)[3]
    ref = tl.tlrmvn_prob(F, w.a, w.b, math.inf, tl.FP64, 2, 100, shifts=w.shifts, per_sample=True)[3]
    assert np.max(np.abs(got - ref) / np.abs(ref)) < 1e-4


@pytest.mark.parametrize("precision", ["FP32", "BF16_SHIFT", "FP16_SHIFT"])
def test_samples_beyond_one_pass(tl, precision):
    M, N = 3, 40031  # 120,093 samples
    w, F = _factor(tl, 150, 70, M, N)
    p = getattr(tl, precision)
    got = tl.tlrmvn_prob(F, w.a, w.b, math.inf, p, M, N, shifts=w.shifts, per_sample=True)[3]
    one = tl.tlrmvn_prob(F, w.a, w.b, math.inf, p, M, N, shifts=w.shifts, per_sample=True, sample_chunk=7000)[3]
    assert np.array_equal(got, one)
