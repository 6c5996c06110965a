"""GPU: the Student-t scale chi_nu^-1(w) / sqrt(nu) against SciPy over the whole range of lattice values. One variable
gives log Phi(b s) per sample, and the shifts put the scale's coordinate at chosen w, from 1e-15 to 1 - 1e-15. Limits
near and far make small and large scales count. Tolerance: the iteration stops within 1e-12 of s, and
log Phi(b s) moves by at most about twice that, relatively, for b < 0."""
import math

import numpy as np
import pytest
from scipy.special import gammainccinv, gammaincinv, log_ndtr

from oracle import lattice

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


def polished(a, x, num):
    """x after a Newton step on P(a, x) = num 2^-53, P by its power series."""
    import mpmath as mp
    with mp.workdps(40):
        A, X = mp.mpf(a), mp.mpf(float(x))
        pref = mp.exp(A * mp.log(X) - X - mp.loggamma(A))
        term, total, k = 1 / A, 1 / A, 0
        while term > total * mp.mpf(10) ** -30:
            k += 1
            term *= X / (A + k)
            total += term
        return float(X - (pref * total - mp.mpf(num) / 2 ** 53) * X / pref)


@pytest.mark.parametrize("nu", [0.5, 1.0, 2.5, 3.0, 3.5, 4.0, 5.0, 7.0, 10.0, 30.0, 1000.0, 1.0e6])
def test_scale(tl, nu):
    tail = 10.0 ** np.linspace(-15.0, -0.302, 6000)
    num = np.round(np.concatenate([tail, 1.0 - tail]) * 2.0 ** 53).astype(np.int64) | 1
    w, wc = num * 2.0 ** -53, (2 ** 53 - num) * 2.0 ** -53
    Q = [int(q) for q in lattice.richtmyer_generators(2)]
    # the point's coordinate x with 2 (x >> 11) + 1 - 2^53 = num, from its shift: x = Q + D
    x = [((int(t) + 2 ** 53 - 1) // 2) << 11 for t in num]
    shifts = np.zeros((len(x), 2), dtype=np.uint64)
    shifts[:, 1] = [(t - Q[1]) % 2 ** 64 for t in x]
    s2 = np.where(w < 0.5, gammaincinv(0.5 * nu, w), gammainccinv(0.5 * nu, wc))
    every = 1
    if nu > 1.0e5:  # (SciPy's inverse is off by up to 4e-12 there: a Newton step in 40 digits, at every 300th point)
        every = 300
        s2[::every] = [polished(0.5 * nu, v, int(t)) for v, t in zip(s2[::every], num[::every])]
    s = np.sqrt(2.0 / nu * s2)
    F = tl.tlrmvn_factor_dense(np.array([[1.0]]), None, None, 1, 0.0, 0, 0)
    for b in (-1.0, -100.0, -1.0e4):
        pm = tl.tlrmvn_prob(F, [-np.inf], [b], nu, tl.FP64, len(x), 1, shifts=shifts, per_sample=True)[3]
        want = log_ndtr(b * s)
        assert np.max((np.abs(np.ravel(pm) - want) / np.abs(want))[::every]) < 4e-12
