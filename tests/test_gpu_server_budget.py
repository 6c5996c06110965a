"""GPU: a float32 request whose general scratch fits a server's budget is served, in smaller passes where the split
path's padded operands do not fit in one; the estimate is the direct call's, bit for bit."""
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


def test_float32_request_near_the_budget(tl):
    M, N, m = 4, 2560, 32
    w = synth.small_workload(0, m, 71, n_shifts=M, n_points=N, ragged_n=600)  # 19 tiles: ranks padded to 64 each
    F = tl.tlrmvn_factor_kernel(w.xy, w.kernel, w.params, w.nugget, w.a, w.b, m, 1e-4, 0, 0)
    one = tl.tlrmvn_prob_scratch_bytes(F, tl.FP32, M, N)
    ktot = int(np.tril(tl.tlrmvn_factor_ranks(F), -1).sum())
    # what the request takes beside the operands (limits, shifts, logs; at most 256 bytes off), and the general path's
    budget = 24 * w.n + 8 * (M * (w.n + 1) + 4 + M + M * N) + 256 + 8 * (2 * w.n + 2) + M * N * ((ktot + 2 * m) * 4 + 8)
    assert budget < one  # (the split path in one pass does not fit)
    want = tl.tlrmvn_prob(F, w.a, w.b, math.inf, tl.FP32, M, N, seed=5)
    srv = tl.Server([F], lanes=1, memory_budget=budget)
    assert srv.wait(srv.submit(0, w.a, w.b, math.inf, tl.FP32, M, N, seed=5))[:2] == want[:2]
    assert srv.stats()["peak_bytes"] <= budget
    srv.close()
    srv = tl.Server([F], lanes=1, memory_budget=budget - 1)
    with pytest.raises(tl.TlrmvnError) as e:  # (what did not fit before is refused as before)
        srv.submit(0, w.a, w.b, math.inf, tl.FP32, M, N, seed=5)
    assert e.value.status == tl.E_BUSY
    srv.close()
