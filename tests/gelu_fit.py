"""Generates the polynomial used by the tensor-core path's GeLU epilogue.

GeLU(x) = x Phi(x) with Phi the standard normal CDF (the exact erf form).
The epilogue writes Phi(x) = (1 + tanh(g(x))) / 2, where g(x) =
atanh(2 Phi(x) - 1) is odd and smooth, and approximates g by x P(x^2) with P
a degree-4 polynomial. The coefficients minimise the largest error of
Phi on [0, 8] (Gauss-Newton steps with Lawson reweighting towards the
minimax solution, numpy/scipy); g then increases monotonically for all x, so
tanh saturates to +-1 beyond the fitted range.

The backward's GeLU is computed more exactly (its value is used in fp32):
Phi(a) = 1/2 + a P(a^2) for |a| < SPLIT, Phi(-|a|) = exp(-a^2/2) t R(t) with
t = 1 / (1 + |a| / 2) beyond (erfcx is smooth in t). P and R minimise the largest
error of Phi (Lawson's algorithm); each coefficient is rounded to fp32 and the
rest fitted again to what is left, so that the rounding of the first ones costs
nothing.

On the GPU, tanh is the hardware approximation tanh.approx.f32, whose error
(about 2^-11) dominates the polynomial's (below 2e-6 on Phi): the GeLU
error stays a small fraction of the bf16 rounding that h receives next.

Run:  python tests/gelu_fit.py   (prints the constants the epilogue in
csrc/tc_common.cuh and the backward in csrc/backward.cu hold;
tests/test_gelu_epilogue.py checks them)
"""
import struct

import numpy as np
from scipy.special import erf, erfcx
from scipy.stats import norm

DEG, X_MAX = 4, 8.0


def _phi_err(c, x):
    return 0.5 * np.tanh(x * np.polyval(c[::-1], x * x)) - (norm.cdf(x) - 0.5)


def fit():
    x = np.linspace(1e-4, X_MAX, 40001)
    c = np.zeros(DEG + 1)
    c[0], c[1] = np.sqrt(2.0 / np.pi), 0.0356774  # tanh-form starting point
    w = np.ones_like(x)
    for _ in range(300):
        e = _phi_err(c, x)
        u = x * x
        t = np.tanh(x * np.polyval(c[::-1], u))
        jac = np.stack([0.5 * (1.0 - t * t) * x * u ** k for k in range(DEG + 1)], 1)
        sw = np.sqrt(w)
        c = c + 0.5 * np.linalg.lstsq(jac * sw[:, None], -e * sw, rcond=None)[0]
        e = _phi_err(c, x)
        w = w * (np.abs(e) / np.abs(e).max() + 1e-3)
        w /= w.mean()
    return c.astype(np.float32)


def gelu_fp32(x, coef):
    """The epilogue's arithmetic in fp32, with an exact tanh."""
    x = x.astype(np.float32)
    u = x * x
    r = np.full_like(u, coef[-1])
    for c in coef[-2::-1]:
        r = (r * u + c).astype(np.float32)
    g = (x * r).astype(np.float32)
    hx = np.float32(0.5) * x
    return (hx * np.tanh(g).astype(np.float32) + hx).astype(np.float32)


SPLIT, P_DEG, R_DEG = 1.35, 5, 3


def _lawson(x, y, w, deg, iters=150):
    """Power-basis coefficients of the polynomial of least max w |P - y|."""
    lo, hi = x.min(), x.max()
    v = np.polynomial.chebyshev.chebvander(2 * (x - lo) / (hi - lo) - 1, deg)
    lw, best = np.ones_like(x), None
    for _ in range(iters):
        sw = np.sqrt(lw) * w
        c = np.linalg.lstsq(v * sw[:, None], y * sw, rcond=None)[0]
        e = w * np.abs(v @ c - y)
        if best is None or e.max() < best[0]:
            best = e.max(), c
        lw = lw * (e / e.max() + 1e-6)
        lw /= lw.mean()
    cheb = np.polynomial.chebyshev.Chebyshev(best[1], domain=[lo, hi])
    return cheb.convert(kind=np.polynomial.Polynomial).coef


def _fit_rounded(x, y, w, deg):
    out = []
    for k in range(deg + 1):
        c0 = np.float64(np.float32(_lawson(x, y, w, deg - k)[0]))
        out.append(c0)
        y, w = (y - c0) / x, w * x
    return np.array(out)


def fit_backward():
    """P and R, lowest coefficient first."""
    u = np.maximum((np.cos(np.linspace(0, np.pi, 2001)) * 0.5 + 0.5) * SPLIT ** 2, 1e-4)
    a = np.sqrt(u)
    p = _fit_rounded(u, 0.5 * erf(a / np.sqrt(2)) / a, a, P_DEG)
    b = np.linspace(SPLIT * 0.995, 9, 4001)[::-1]
    t = 1 / (1 + 0.5 * b)
    r = _fit_rounded(t, 0.5 * erfcx(b / np.sqrt(2)) / t, (np.exp(-b * b / 2) + 1e-7) * t, R_DEG)
    return p, r


def phi_backward(a, p, r):
    """The backward's Phi in fp32 (fused multiply-adds rounded once), with exact
    exponential and reciprocal."""
    f32, f64 = np.float32, np.float64
    a = a.astype(f32)
    u = a * a

    def horner(c, x):
        v = np.full_like(x, f32(c[-1]))
        for k in c[-2::-1]:
            v = (v.astype(f64) * x + f64(f32(k))).astype(f32)
        return v

    e = np.exp2((u * f32(-0.72134752044448170)).astype(f64)).astype(f32)
    t = (1 / (np.abs(a).astype(f64) * 0.5 + 1).astype(f32).astype(f64)).astype(f32)
    near = (a.astype(f64) * horner(p, u) + 0.5).astype(f32)
    q = np.copysign(horner(r, t) * t, a)
    far = ((a > 0) - q.astype(f64) * e).astype(f32)
    return np.where(np.abs(a) < f32(SPLIT), near, far)


if __name__ == "__main__":
    coef = fit()
    x = np.linspace(-12, 12, 480001)
    ref = x * norm.cdf(x)
    g = gelu_fp32(x, coef).astype(np.float64)
    phi_err = np.abs(_phi_err(coef.astype(np.float64), np.linspace(1e-4, X_MAX, 40001))).max()
    gg = np.linspace(0, 1e3, 100001)
    mono = bool(np.all(np.diff(gg * np.polyval(coef[::-1].astype(np.float64), gg * gg)) > 0))
    print("// max |Phi err| %.2e, max |GeLU err| / max(|x|, 1) %.2e, g monotone: %s"
          % (phi_err, (np.abs(g - ref) / np.maximum(np.abs(x), 1)).max(), mono))
    for i, c in enumerate(coef):
        bits = struct.unpack("<I", struct.pack("<f", float(c)))[0]
        print("  0x%08x  // c%d = %.9g" % (bits, i, c))
    p, r = fit_backward()
    print("// backward: P", ", ".join("%.9g" % c for c in p))
    print("// backward: R", ", ".join("%.9g" % c for c in r))
