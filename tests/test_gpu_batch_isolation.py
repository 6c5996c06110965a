"""GPU: one problem of a batched plan whose numbers are not finite (limits 1e20 standard deviations out, a NaN in its
factor) beside an ordinary one: the ordinary one's estimate is that of other runs, in the same run (about
twice as many items as blocks: blocks go from one problem to the other) and in later ones. BF16: bit for bit. FP32: a
run beyond fp16's range is repeated by the general kernel, 1e-6 relative."""
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


@pytest.mark.parametrize("precision", ["FP32", "BF16_SHIFT"])
@pytest.mark.parametrize("cause", ["limits", "B", "V"])
def test_neighbour_unharmed(tl, precision, cause):
    # tiles of 100 and 70: the second problem's padding rows and columns lie where the first one's values were
    ws = [synth.small_workload(0, m, 330 + m, ragged_n=n) for n, m in ((300, 100), (280, 70))]
    Fs = [tl.tlrmvn_factor_kernel(w.xy, w.kernel, w.params, w.nugget, w.a, w.b, w.m, w.tol, 0, 0) for w in ws]
    p = getattr(tl, precision)
    a, b = [w.a for w in ws], [w.b for w in ws]
    bad = [b[0].copy(), b[1]]
    if cause == "limits":
        bad[0][::3] = -1.0e20
    else:
        ex = tl.parse_export(tl.tlrmvn_factor_export(Fs[0]))
        sizes = np.diff(ex.tile_off)
        B = [ex.B[t, :sizes[t], :sizes[t]].copy() for t in range(ex.r)]
        if cause == "B":
            B[0][70, 3] = np.nan
        else:
            ex.V[(1, 0)][5, 0] = np.nan
        broken = tl.tlrmvn_factor_import(tl.build_export(ex.n, ex.m, ex.tile_off, ex.perm, B, ex.U, ex.V))
    ok = tl.BatchPlan(Fs, math.inf, 2, 128 * 950, seed=9, precision=p)
    first = ok.run(a, b)[0]
    plan = ok if cause == "limits" else tl.BatchPlan([broken, Fs[1]], math.inf, 2, 128 * 950, seed=9, precision=p)
    for _ in range(3):
        got = plan.run(a, bad)[0]
        assert not np.isfinite(got[0])
        assert got[1] == first[1] if precision == "BF16_SHIFT" else abs(got[1] - first[1]) < 1e-6 * abs(first[1])
        assert np.array_equal(ok.run(a, b)[0], first)
    plan.close()
    ok.close()
