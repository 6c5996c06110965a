"""GPU: limits beyond fp16's range on the FP16-shift path (a y or a projection above 65,504 in size): the solve is
repeated in float32, so the samples match the oracle's within the float32 path's 1e-4 relative, with any number of
samples per pass."""
import math

import numpy as np
import pytest

import synth
from oracle import sov
from tests.helpers import export_bytes, oracle_factor

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


@pytest.mark.parametrize("far", [-6.0e4, -1.0e5, -2.0e6])
@pytest.mark.parametrize("limits", ["uniform", "twosided"])
def test_fp16_range(tl, far, limits):
    w = synth.small_workload(0, 100, 321, n_shifts=2, n_points=130, ragged_n=250, limits=limits)
    OF, _ = oracle_factor(w)
    F = tl.tlrmvn_factor_import(export_bytes(OF))
    a, b = w.a.copy(), w.b.copy()
    a[::40], b[::40] = (-np.inf if limits == "uniform" else 1.001 * far), far
    ref = sov.solve(OF, a, b, math.inf, w.shifts, w.n_points)["per_sample"]
    for chunk in (0, 256):
        pm = tl.tlrmvn_prob(F, a, b, math.inf, tl.FP16_SHIFT, 2, 130, shifts=w.shifts, per_sample=True,
                            sample_chunk=chunk)[3]
        assert np.max(np.abs(pm - ref) / np.abs(ref)) < 1e-4


def test_large_limits_within_range(tl):
    # y up to 60,000: still the fp16 products
    w = synth.small_workload(0, 64, 322, n_shifts=2, n_points=130, ragged_n=150)
    OF, _ = oracle_factor(w)
    F = tl.tlrmvn_factor_import(export_bytes(OF))
    b = w.b.copy()
    b[::40] = -3.0e4
    ref = sov.solve(OF, w.a, b, math.inf, w.shifts, w.n_points)["per_sample"]
    pm = tl.tlrmvn_prob(F, w.a, b, math.inf, tl.FP16_SHIFT, 2, 130, shifts=w.shifts, per_sample=True)[3]
    assert np.max(np.abs(pm - ref) / np.abs(ref)) < 1e-2
