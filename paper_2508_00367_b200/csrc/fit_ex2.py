"""Fits the polynomial of the attention kernel's 2^x on the FMA pipes (rs_attn.cuh, ex2_pair_fma).

2^x = 2^n * 2^f with n = round(x) and f in [-1/2, 1/2].  A degree-5 polynomial is fitted to 2^f by iteratively re-weighted
least squares (Lawson) under the weight 2^-f, i.e. for the least maximum relative error, and the whole function is checked
in emulated fp32 arithmetic (fused multiply-adds: one rounding of the exact product and sum).

    python fit_ex2.py        # prints the coefficients (lowest degree first) and the max relative error
"""
import numpy as np


def fit(deg=5, iters=200):
    f = np.linspace(-0.5, 0.5, 20001)
    w = np.exp2(-f)
    lam = np.ones_like(f)
    V = np.vander(f, deg + 1, increasing=True)
    coef = None
    for _ in range(iters):
        ww = w * np.sqrt(lam)
        coef, *_ = np.linalg.lstsq(V * ww[:, None], np.exp2(f) * ww, rcond=None)
        r = np.abs((V @ coef - np.exp2(f)) * w)
        lam = lam * (r / r.max() + 1e-3)
        lam /= lam.mean()
    return coef


def ex2_fp32(x, coef):
    """The kernel's steps on fp32 values x <= 120 (fp64 holds a product of two fp32 values exactly)."""
    c = np.asarray(coef).astype(np.float32)
    with np.errstate(invalid="ignore"):
        x = np.where(np.isnan(x), x, np.maximum(x, np.float32(-127.0))).astype(np.float32)
    n = np.rint(x)
    f = (x - n).astype(np.float32)
    q = np.full_like(x, c[-1])
    for ci in c[-2::-1]:
        q = (q.astype(np.float64) * f + ci).astype(np.float32)
    scale = np.where(n > -127, np.exp2(np.nan_to_num(n).astype(np.float64)), 0.0).astype(np.float32)
    return (q * scale).astype(np.float32)


def max_rel_error_fp32(coef, lo=-125.0, hi=8.0, n=2000001):
    x = np.linspace(lo, hi, n).astype(np.float32)
    ref = np.exp2(x.astype(np.float64))
    return float((np.abs(ex2_fp32(x, coef) - ref) / ref).max())


if __name__ == "__main__":
    c = fit()
    print([float(np.float32(v)) for v in c])
    print("max relative error of 2^x in fp32: %.3e" % max_rel_error_fp32(c))
