"""GPU: launch choices on the paths that they still reach. The general float32 sweep (sub-tile, block size, samples
per pass) runs after a y beyond fp16's range: here the last variable's, alone in its tile and independent of the
others, so that its constant log can be taken off; every choice matches the oracle on the other 512 within 1e-4
relative per sample. The whole-tile sweep's CTAs per SM count from more than two of them: the same bits for each choice."""
import math

import numpy as np
import pytest

import synth
from oracle import sov
from tests.helpers import oracle_factor

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


def far_factor(tl, OF):
    U = {k: u for k, u in OF.U.items() if u.shape[1]}
    return tl.tlrmvn_factor_import(tl.build_export(OF.n + 1, OF.m, np.append(OF.tile_off, OF.n + 1),
                                                   np.append(OF.perm, OF.n), [*OF.B, np.eye(1)], U,
                                                   {k: OF.V[k] for k in U}))


@pytest.mark.parametrize("limits", ["uniform", "twosided"])
def test_general_float32_choices(tl, limits):
    n, M, N = 512, 3, 500
    w = synth.small_workload(0, 256, 64, n_shifts=M, n_points=N, ragged_n=n, limits=limits)
    OF, _ = oracle_factor(w)
    F = far_factor(tl, OF)
    ref = np.ravel(sov.solve(OF, w.a, w.b, math.inf, w.shifts, N)["per_sample"])
    shifts = np.concatenate([w.shifts, w.shifts[:, :1]], axis=1)
    a, b = np.append(w.a, -np.inf if limits == "uniform" else -1.0e5), np.append(w.b, -5.0e4)
    for sub in (64, 128):
        for threads in (0, 64, 128, 256):
            for chunk in (0, 512):
                tl.tlrmvn_set_tuning(F, tl.FP32, sub=sub, threads=threads, chunk=chunk)
                pm = np.ravel(tl.tlrmvn_prob(F, a, b, math.inf, tl.FP32, M, N, shifts=shifts, per_sample=True)[3])
                d = pm - ref  # the far variable's log, -1.25e9, plus the others' errors
                assert abs(np.median(d) + 1.25e9) < 1e3
                # (-1.25e9 is a multiple of 2^-22 in float64)
                assert np.max(np.abs(d - np.median(d)) / np.abs(ref)) < 1e-4, (sub, threads, chunk)


@pytest.mark.parametrize("precision", ["BF16_SHIFT", "FP16_SHIFT", "FP32"])
def test_ctas_per_sm(tl, precision):
    M, N = 4, 10240  # 320 blocks: more than two an SM
    p = getattr(tl, precision)
    w = synth.small_workload(0, 70, 65, nu=3.0, n_shifts=M, n_points=N, ragged_n=150)
    F = tl.tlrmvn_factor_kernel(w.xy, w.kernel, w.params, w.nugget, w.a, w.b, w.m, w.tol, 0, 0)
    kw = dict(n_shifts=M, n_points=N, shifts=w.shifts, per_sample=True)
    base = tl.tlrmvn_prob(F, w.a, w.b, w.nu, p, **kw)[3]
    for ctas in (4, 2, 1):
        tl.tlrmvn_set_tuning(F, p, tc_ctas=ctas)
        assert np.array_equal(tl.tlrmvn_prob(F, w.a, w.b, w.nu, p, **kw)[3], base), ctas
    ref = tl.tlrmvn_prob(F, w.a, w.b, w.nu, tl.FP64, **kw)[3]
    assert np.max(np.abs(base - ref) / np.abs(ref)) < (1e-4 if precision == "FP32" else 1e-2)
