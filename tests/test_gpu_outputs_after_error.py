"""GPU: the estimator's outputs after a solve whose kernels recorded an error stay as they were: the bounded wait's
self-test runs the estimator behind a wait that gave up and compares the outputs' bytes (a change is TLRMVN_E_CUDA);
a call refused for its limits leaves device outputs alone too."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def test_outputs_left_alone():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__ as ge
    ge.build()
    import paper_2003_11183_gb300 as tl
    from paper_2003_11183_gb300 import _lib
    assert tl.tlrmvn_selftest_wait_timeout(100) == tl.E_TIMEOUT
    assert "estimate" not in _lib.load().tlrmvn_last_error().decode()
    F = tl.tlrmvn_factor_dense(np.eye(4), None, None, 4, 1e-9, 0, 0)
    out = torch.full((2,), 7.0, dtype=torch.float64, device="cuda")
    a = torch.full((4,), math.nan, dtype=torch.float64, device="cuda")
    with pytest.raises(tl.TlrmvnError):
        tl.tlrmvn_prob_device(F, a, a, out, math.inf, tl.BF16_SHIFT, 2, 100)
    assert out.tolist() == [7.0, 7.0]
