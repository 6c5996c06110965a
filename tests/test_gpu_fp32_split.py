"""GPU: the float32 path on split fp16 operands (STC_FP32 in csrc/sweep_tc.cuh) where it can go wrong: tiles at the
edges of the 64-variable sub-tile and of the 128-sample block, rows of very different scale (a power of two each),
and y beyond fp16's range (repeated by the general float32 integrand, single and batched).  Tolerance: the float32
path's 1e-4 relative per sample, as on every other problem."""
import math

import numpy as np
import pytest

import synth
from oracle import sov
from tests.helpers import export_bytes, oracle_factor, to_oracle_factor

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


def rel(a, b):
    return np.max(np.abs(np.asarray(a) - np.asarray(b)) / np.abs(np.asarray(b)))


@pytest.mark.parametrize("n,m,M,N", [(5, 1, 1, 1), (70, 7, 3, 43), (129, 63, 2, 64), (130, 64, 1, 127), (200, 65, 3, 43),
                                     (300, 130, 2, 129), (257, 256, 1, 300)])
@pytest.mark.parametrize("limits,nu", [("uniform", math.inf), ("twosided", 3.0)])
def test_edges(tl, n, m, M, N, limits, nu):
    w = synth.small_workload(0, m, 300 + n, nu=nu, n_shifts=M, n_points=N, ragged_n=n, limits=limits)
    OF, _ = oracle_factor(w)
    F = tl.tlrmvn_factor_import(export_bytes(OF))
    pm = tl.tlrmvn_prob(F, w.a, w.b, nu, tl.FP32, M, N, shifts=w.shifts, per_sample=True)[3]
    assert rel(pm, sov.solve(OF, w.a, w.b, nu, w.shifts, N)["per_sample"]) < 1e-4


def test_rows_of_different_scale(tl):
    from oracle import geometry
    w = synth.small_workload(0, 128, 310, n_shifts=2, n_points=200, ragged_n=500, tol=1e-9)
    d = 10.0 ** np.random.default_rng(3).uniform(-3.0, 3.0, w.n)
    Sig = geometry.covariance(w.xy, w.kernel, w.params, w.nugget) * d[:, None] * d[None, :]
    F = tl.tlrmvn_factor_dense(Sig, None, None, 128, 1e-9, 0, 0)
    OF = to_oracle_factor(tl.parse_export(tl.tlrmvn_factor_export(F)))
    ref = sov.solve(OF, w.a, w.b * d, math.inf, w.shifts, w.n_points)
    pm = tl.tlrmvn_prob(F, w.a, w.b * d, math.inf, tl.FP32, 2, 200, shifts=w.shifts, per_sample=True)[3]
    assert rel(pm, ref["per_sample"]) < 1e-4


def test_y_beyond_fp16_range(tl):
    # limits 50,000 and 2e6 standard deviations out: y of that size, and finite results
    w = synth.small_workload(0, 64, 320, n_shifts=2, n_points=130, ragged_n=150)
    OF, _ = oracle_factor(w)
    F = tl.tlrmvn_factor_import(export_bytes(OF))
    for far in (-5.0e4, -2.0e6):
        b = w.b.copy()
        b[::40] = far
        ref = sov.solve(OF, w.a, b, math.inf, w.shifts, w.n_points)
        lp, _, _, pm = tl.tlrmvn_prob(F, w.a, b, math.inf, tl.FP32, 2, 130, shifts=w.shifts, per_sample=True)
        assert rel(pm, ref["per_sample"]) < 1e-4
        plan = tl.BatchPlan([F, F], math.inf, 2, 130, seed=7)
        one = [tl.tlrmvn_prob(F, w.a, b, math.inf, tl.FP32, 2, 130, seed=7 + p)[0] for p in range(2)]
        assert rel(plan.run([w.a] * 2, [b] * 2)[0], one) < 1e-4
        near = plan.run([w.a] * 2, [w.b] * 2)[0]  # the plan's usual kernel again
        one = [tl.tlrmvn_prob(F, w.a, w.b, math.inf, tl.FP32, 2, 130, seed=7 + p)[0] for p in range(2)]
        assert rel(near, one) < 1e-6
        plan.close()


def test_batch_after_values_beyond_range(tl):
    # a plan whose blocks serve a problem of larger tiles with y beyond fp16's range in one run and one of smaller tiles in
    # the next: what the first left in the blocks' buffers (the smaller one's padding) must not reach it, nor what
    # invalid limits left.  (About as many items as blocks, so that blocks change problems from run to run.)
    M, N = 2, 12800
    ws = [synth.small_workload(0, m, 330 + m, ragged_n=n) for n, m in ((300, 100), (280, 70))]
    Fs = [tl.tlrmvn_factor_kernel(w.xy, w.kernel, w.params, w.nugget, w.a, w.b, w.m, w.tol, 0, 0) for w in ws]
    plan = tl.BatchPlan(Fs, math.inf, M, N, seed=9)
    a, b = [w.a for w in ws], [w.b for w in ws]
    first = plan.run(a, b)[0]
    far, nan = b[0].copy(), b[0].copy()
    far[::3] = -2.0e6
    nan[::7] = np.nan
    for _ in range(8):
        plan.run(a, [far, b[1]])
        assert rel(plan.run(a, b)[0], first) < 1e-6
        with pytest.raises(tl.TlrmvnError):
            plan.run(a, [nan, b[1]])
        assert rel(plan.run(a, b)[0], first) < 1e-6
    plan.close()
