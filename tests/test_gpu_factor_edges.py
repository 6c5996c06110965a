"""GPU: the factorisation at the edges of its kernels' tiles against the oracle: blocks around the 64-wide Cholesky
panel and the 16-wide product groups, clusters of eight CTAs with ragged or no rows in some (tiles of 1 to 33;
past 430 one CTA), a short last tile, two-sided limits and limits far above the tables of the conditioning's probabilities.  Orders and ranks
equal, the dense factor within 1e-7 (truncation at 1e-9)."""
import numpy as np
import pytest

import synth
from tests.helpers import oracle_factor, to_oracle_factor

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


CASES = [(nm, rl) for nm in [(9, 1), (20, 7), (70, 33), (129, 64), (131, 65), (200, 100), (300, 150)]
         for rl in [(0, "uniform"), (1, "uniform"), (2, "uniform"), (2, "twosided"), (2, "high")]]
CASES.append(((900, 450), (1, "uniform")))  # a tile whose residual does not fit the cluster's shared memory


@pytest.mark.parametrize("nm,rl", CASES)
def test_factor_edges(tl, nm, rl):
    (n, m), (reorder, limits) = nm, rl
    w = synth.small_workload(0, m, 400 + n, ragged_n=n, tol=1e-9, reorder=reorder,
                             limits="uniform" if limits == "high" else limits)
    if limits == "high":  # probabilities that round to 1, some limits beyond 13 standard deviations
        w.b[:] = np.random.default_rng(n).uniform(4.0, 15.0, n)
    OF, _ = oracle_factor(w)
    F = tl.tlrmvn_factor_kernel(w.xy, w.kernel, w.params, w.nugget, w.a, w.b, m, w.tol, 0, reorder)
    ex = tl.parse_export(tl.tlrmvn_factor_export(F))
    assert np.array_equal(ex.perm, OF.perm) and np.array_equal(ex.tile_off, OF.tile_off)
    assert np.abs(to_oracle_factor(ex).dense() - OF.dense()).max() < 1e-7
