"""Coefficients of phi_neg_f32 in sov_device.cuh (run to reproduce them).

Phi(-x) = exp(-x^2/2) R(x) with R(x) = erfcx(x/sqrt(2)) / 2, fitted on [0, 13] as a
degree-9 polynomial in 1 / (2.5 + x) with the smallest maximum relative error (Lawson's
iteratively reweighted least squares; 6.2e-8 in float64).  In float32, its even and odd
halves evaluated side by side, the relative error is 4.0e-7 at most and 8e-8 rms
(exact 2^f and reciprocal).
"""
import numpy as np
from scipy.special import erfcx


def lawson(a: np.ndarray, y: np.ndarray, steps: int = 300) -> np.ndarray:
    """Coefficients c with the smallest maximum of |a c / y - 1|."""
    lam, best = np.ones(len(y)), (np.inf, None)
    for _ in range(steps):
        w = np.sqrt(lam) / np.abs(y)
        c = np.linalg.lstsq(a * w[:, None], y * w, rcond=None)[0]
        e = np.abs(a @ c / y - 1.0)
        if e.max() < best[0]:
            best = (e.max(), c)
        lam = lam * e
        lam = np.maximum(lam / lam.sum(), 1e-18)
    return best[1]


def fit(deg: int = 9, c: float = 2.5, top: float = 13.0, points: int = 8000) -> np.ndarray:
    x = (1.0 - np.cos(np.linspace(0.0, np.pi, points))) / 2.0 * top
    r = 0.5 * erfcx(x / np.sqrt(2))
    t = 1.0 / (c + x)
    lo, hi = t.min(), t.max()
    co = lawson(np.polynomial.chebyshev.chebvander((2.0 * t - lo - hi) / (hi - lo), deg), r)
    return np.polynomial.Chebyshev(co, domain=[lo, hi]).convert(kind=np.polynomial.Polynomial).coef


if __name__ == "__main__":
    co = fit()
    x = np.linspace(0.0, 13.0, 100001)
    r = 0.5 * erfcx(x / np.sqrt(2))
    print("max relative error (float64):", np.max(np.abs(np.polyval(co[::-1], 1.0 / (2.5 + x)) / r - 1)))
    print(", ".join(f"{c:.9e}f" for c in co.astype(np.float32)))
