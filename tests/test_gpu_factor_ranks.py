"""GPU: the ranks that the factorisation finds, tile by tile, equal the oracle's, uncapped and capped, with the exact and
the tile-low-rank Schur complement, in clusters of eight CTAs and (tiles past some 430) by one. With equal ranks and both
residuals within the tolerance the dense factors differ by a few tolerances (twenty allowed: tiles of earlier columns enter
the later ones)."""
import numpy as np
import pytest

import synth
from oracle import factor as ofactor, geometry
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


CASES = [(*size, reorder, schur) for size in [(70, 33, 1e-9, 0), (131, 65, 1e-6, 0), (300, 70, 1e-4, 0), (400, 100, 1e-6, 5),
                                              (300, 150, 1e-9, 12)] for reorder in (0, 1, 2) for schur in (0, 1)]
CASES.append((900, 450, 1e-6, 0, 1, 0))


@pytest.mark.parametrize("n,m,tol,cap,reorder,schur", CASES)
def test_ranks(tl, n, m, tol, cap, reorder, schur):
    w = synth.small_workload(0, m, 600 + n, ragged_n=n, tol=tol, max_rank=cap, reorder=reorder)
    if schur:
        perm0, sizes = geometry.kd_order(w.xy, m)
        Sig = geometry.covariance(w.xy, w.kernel, w.params, w.nugget)
        OF = ofactor.tlr_factor_truncated(Sig, perm0, sizes, w.a, w.b, tol, cap or m, reorder)
    else:
        OF, _ = oracle_factor(w)
    F = tl.tlrmvn_factor_kernel(w.xy, w.kernel, w.params, w.nugget, w.a, w.b, m, tol, cap, reorder, schur=schur)
    ex = tl.parse_export(tl.tlrmvn_factor_export(F))
    GF = to_oracle_factor(ex)
    assert np.array_equal(ex.perm, OF.perm)
    assert {k: u.shape[1] for k, u in GF.U.items()} == {k: u.shape[1] for k, u in OF.U.items()}
    assert tl.tlrmvn_factor_info(F)["capped"] == OF.capped_tiles
    assert np.abs(GF.dense() - OF.dense()).max() < (20 * tol if not cap else 1e-7)
