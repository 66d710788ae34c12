"""Writes core_fit.cuh: the polynomial pieces of the Gaussian core used by the
FP32 near-field kernel.

K(r; a) of Eq. vem1 with x = r/a, u = x^2:

* x < 1.5 (u < 2.25): F(u) = K/x^3 and its derivative F'(u).  Since
  dK/dx = sqrt(2/pi) x^2 exp(-x^2/2), integrating the exponential series term by
  term gives F(u) = sqrt(2/pi) sum_k (-1)^k u^k / (2^k k! (2k+3)), which has no
  cancellation at small x.  F' is interpolated at the Chebyshev nodes of [0, 2.25]
  (degree 7) and written as a polynomial in s = (2u - 2.25)/2.25, without the factor
  sqrt(2/pi) (it sits in the kernel's constants); the same equation gives
  F = (exp(-u/2) - 2 u F') / 3, a sum of positive terms (F' < 0).
* 1.5 <= x < 6.5: 1 - K = exp(-u/2) x G(y), y = 1/x,
  G(y) = y exp(x^2/2) erfc(x/sqrt 2) + sqrt(2/pi), smooth in y, as a polynomial in
  t = (2y - (1/1.5 + 1/6.5)) / (1/1.5 - 1/6.5), so that f K = f - (exp(-u/2) / (a r^2)) G takes
  no separate r.  An error of G enters the relative errors of K / r^3 and of its derivative term
  with the weights x exp(-x^2/2) / K and exp(-x^2/2) / (x^2 (K/x^3 - sqrt(2/pi) exp(-x^2/2) / 3)), 1.0
  and 2.6 at x = 1.5 and below 1e-8 at 6.5, and those enter the velocity of a uniform cloud with
  K / x^2 and the volume x^2 dx: G is the weighted least-squares polynomial of degree 5.

The kernel takes the coefficients with the powers of a that its pieces carry (CoreConsts).
Reference values are 40-digit mpmath; the header reports the maximal errors.
Run: python gen_core_fit.py  (needs mpmath; the header is committed).
"""
import os

import mpmath as mp
import numpy as np

U_HI = 2.25
Y_LO, Y_HI = 1 / 6.5, 1 / 1.5
DEG_S, DEG_G = 7, 5


def Fp(u):
    u = mp.mpf(u)
    return mp.nsum(lambda k: (-1) ** k * k * u ** (k - 1) / (2 ** k * mp.factorial(k) * (2 * k + 3)), [1, mp.inf])


def E(y):
    """exp(x^2/2) erfc(x/sqrt 2) at x = 1/y."""
    x = 1 / mp.mpf(y)
    return mp.e ** (x * x / 2) * mp.erfc(x / mp.sqrt(2))


def G(y):
    """y E(y) + sqrt(2/pi): R(x) = G(y) x at y = 1/x."""
    y = mp.mpf(y)
    return y * E(y) + mp.sqrt(2 / mp.pi)


def fit(fun, lo, hi, deg):
    k = np.arange(deg + 1)
    tn = np.cos(np.pi * (k + 0.5) / (deg + 1))
    xn = (tn * (hi - lo) + (hi + lo)) / 2
    cheb = np.polynomial.chebyshev.chebfit(tn, np.array([float(fun(x)) for x in xn]), deg)
    mono = np.polynomial.chebyshev.cheb2poly(cheb)
    tt = np.linspace(-1, 1, 1601)
    xx = (tt * (hi - lo) + (hi + lo)) / 2
    ref = np.array([float(fun(x)) for x in xx])
    err = float(np.max(np.abs(np.polynomial.polynomial.polyval(tt, mono.astype(np.float32)) - ref) / np.abs(ref)))
    return mono, err


def fit_weighted_G(deg):
    """Monomials in t of the degree-`deg` weighted least-squares polynomial of G on y in [Y_LO, Y_HI]
    (weights: see above), and the largest and the weighted rms errors in f and g when it is evaluated
    in FP32 (fused multiply-adds, t from the rounded y as the kernel forms it)."""
    x = np.linspace(1 / Y_HI, 1 / Y_LO, 2001)
    y = 1 / x
    g = np.array([float(G(v)) for v in y])
    e = np.exp(-x * x / 2)
    k = 1 - e * g * x
    wf = x * e / k
    wg = e / x ** 2 / (k / x ** 3 - np.sqrt(2 / np.pi) / 3 * e)
    dens = (k / x) ** 2
    t = (2 * y - (Y_HI + Y_LO)) / (Y_HI - Y_LO)
    cheb = np.polynomial.chebyshev.chebfit(t, g, deg, w=np.sqrt(dens) * np.maximum(wf, wg))
    mono = np.polynomial.chebyshev.cheb2poly(cheb)
    f32 = lambda a: np.asarray(a).astype(np.float32).astype(np.float64)  # noqa: E731
    tf = f32(f32(y) * (2 / (Y_HI - Y_LO)) - (Y_HI + Y_LO) / (Y_HI - Y_LO))
    p = np.full_like(tf, f32(mono[-1]))
    for q in mono[-2::-1]:
        p = f32(p * tf + f32(q))
    rms = lambda w: float(np.sqrt(np.sum(dens * (w * (p - g)) ** 2) / np.sum(dens)))  # noqa: E731
    return mono, float(np.max(wf * np.abs(p - g))), float(np.max(wg * np.abs(p - g))), rms(wf), rms(wg)


def main():
    mp.mp.dps = 40
    fps, efp = fit(Fp, 0.0, U_HI, DEG_S)
    fg, egf, egg, rgf, rgg = fit_weighted_G(DEG_G)
    lines = [
        "// Generated by gen_core_fit.py -- do not edit.",
        "// Gaussian core of Eq. vem1, x = r/a, u = x^2 (the packed FP32 near-field kernel; host arrays,",
        "// the kernel gets them with their powers of a).",
        f"// x < 1.5: d(K/x^3)/du = sqrt(2/pi) sum_k kSerFp[k] s^k, s = (2u - {U_HI})/{U_HI}; max rel.",
        f"//   error {efp:.1e} (coefficients in FP32); K/x^3 = (sqrt(2/pi) exp(-u/2) - 2u d(K/x^3)/du) / 3.",
        "// 1.5 <= x < 6.5: 1 - K = exp(-u/2) x G(y), G = sum_k kCoreFitG[k] t^k, y = 1/x,",
        f"//   t = (2y - {Y_HI + Y_LO:.17g})/{Y_HI - Y_LO:.17g}; evaluated in FP32 the error of G",
        f"//   makes at most {egf:.1e} (rms {rgf:.1e}) of K/r^3 and {egg:.1e} ({rgg:.1e}) of its derivative term.",
        "#pragma once",
        f"#define LHV_CORE_SER_DEG {DEG_S}",
        f"#define LHV_CORE_G_DEG {DEG_G}",
        f"#define LHV_CORE_U_SER {U_HI}f",
        f"#define LHV_CORE_Y_SCALE {2 / (Y_HI - Y_LO):.9e}f",
        f"#define LHV_CORE_Y_SHIFT {-(Y_HI + Y_LO) / (Y_HI - Y_LO):.9e}f",
    ]
    for name, arr in (("kSerFp", fps), ("kCoreFitG", fg)):
        lines.append(f"static const double {name}[{len(arr)}] = {{")
        lines += [f"    {c:.17e}," for c in arr]
        lines.append("};")
    lines.append("")
    out = os.path.join(os.path.dirname(os.path.abspath(__file__)), "core_fit.cuh")
    with open(out, "w") as f:
        f.write("\n".join(lines))
    print(out, efp, egf, egg, rgf, rgg)


if __name__ == "__main__":
    main()
