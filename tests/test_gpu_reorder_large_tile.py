"""GPU: the within-tile reordering of imported tiles whose conditioning leaves no room for its tables in shared memory
(from 3,184 variables; the largest that the inverses take is 3,632). Independent variables: the order is that of
the limits."""
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


@pytest.mark.parametrize("n", [2700, 3184, 3632])
def test_large_tile(tl, n):
    F = tl.tlrmvn_factor_import(tl.build_export(n, n, np.array([0, n]), np.arange(n), [np.eye(n)], {}, {}))
    b = np.random.default_rng(n).permutation(np.linspace(-6.0, 14.0, n))
    G = tl.tlrmvn_factor_reorder_tiles(F, np.full(n, -np.inf), b)
    assert np.array_equal(tl.parse_export(tl.tlrmvn_factor_export(G)).perm, np.argsort(b))
