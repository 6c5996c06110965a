"""Coefficients of the central region of ndtri_f32 in common.cuh (run to reproduce them).

For p in (0, 1/2], L = log2(4 p (1 - p)) (the variable M. Giles uses for the inverse
error function, "Approximating the erfinv function", GPU Computing Gems, 2011, in the
base of the hardware logarithm) and x = 1 - 2p, Phi^-1(p) = x S(L) with S a smooth
function of L.  For p > 8.4e-5 (L > -8 / ln 2) S is fitted here as a degree-11
polynomial in L + 3 with the smallest maximum relative error (1.4e-8 in float64).  In float32, its even and
odd halves evaluated side by side, the relative error is 2.4e-7 at most and 5e-8 rms (an exact logarithm);
the shift 3 keeps the two halves from cancelling.  The reference values come from
SciPy's float64 normal quantile through p = exp(-w) / (2 (1 + x)), w = -L ln 2, which has no
cancellation.
"""
import numpy as np
from scipy.special import ndtri

from fit_mills import lawson

W_MAX, SHIFT, DEG = 8.0, 3.0, 11


def s_of_w(w: np.ndarray) -> np.ndarray:
    x = np.sqrt(-np.expm1(-w))
    return ndtri(np.exp(-w) / (2.0 * (1.0 + x))) / x


def fit(points: int = 8001) -> np.ndarray:
    w = ((1.0 - np.cos(np.linspace(0.0, np.pi, points))) / 2.0 * W_MAX)[1:]
    top = W_MAX / np.log(2)
    co = lawson(np.polynomial.chebyshev.chebvander(1.0 - 2.0 * w / W_MAX, DEG), s_of_w(w))
    return np.polynomial.Chebyshev(co, domain=[SHIFT - top, SHIFT]).convert(kind=np.polynomial.Polynomial).coef


if __name__ == "__main__":
    co = fit()
    w = np.linspace(0.0, W_MAX, 200001)[1:]
    print("max relative error (float64):", np.max(np.abs(np.polyval(co[::-1], SHIFT - w / np.log(2)) / s_of_w(w) - 1)))
    print(", ".join(f"{c:.9e}f" for c in co.astype(np.float32)))
