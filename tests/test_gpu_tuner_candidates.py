"""GPU: the tuner times the whole-tile sweep's CTAs per SM only where a pass has more than two of them."""
import math

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


@pytest.mark.parametrize("points,candidates", [(500, 2), (10240, 3)])
def test_tuner_candidates(tl, points, candidates):
    # a pass of half the samples has at most two CTAs an SM in both, all samples at once more than two in the second
    w = synth.small_workload(0, 70, 66, n_shifts=4, n_points=points, ragged_n=150)
    F = tl.tlrmvn_factor_kernel(w.xy, w.kernel, w.params, w.nugget, w.a, w.b, w.m, w.tol, 0, 0)
    got = tl.tlrmvn_autotune(F, w.a, w.b, math.inf, tl.BF16_SHIFT, n_shifts=4, n_points=points, shifts=w.shifts)
    assert got["candidates"] == candidates
    if candidates == 2:
        assert got["tc_ctas"] == 6
