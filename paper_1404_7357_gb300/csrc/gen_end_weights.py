"""Writes end_weights.cuh: the endpoint weights of the back-projection's sample sums.

For h band-limited to b in [c - w, c + w] (radians per sample) and samples at the integers,

  int_{-inf}^{f} h(t) / sqrt(f - t) dt = sum_{k <= -m} h(k) / sqrt(f - k) + sum_{j=1-m}^{p} w_j(f) h(j)

with 0 <= f < 1: the trapezoidal rule up to the sample m short of the end's integer part, and
m + p weights (complex, since the band is not symmetric) that depend on f alone.  With h =
exp(-i b t) both sides are linear in w: the weights are the least-squares solution over the band,
A w = C with A_bj = exp(-i b j) and C(b) the windowed integral minus the windowed regular sum (a
smooth window far from the end changes neither).  The matrix does not depend on f, so one
truncated pseudo-inverse serves every f and w_j is as smooth in f as C; each is stored as a
polynomial in x = 2 f - 1.  Corrected trapezoidal rules for an inverse square root singularity
of this kind: Kapur & Rokhlin, SIAM J. Numer. Anal. 34 (1997); Alpert, SIAM J. Sci. Comput. 20
(1999).

Usage: python gen_end_weights.py > end_weights.cuh   (prints the worst error to stderr)
"""
import math
import sys

import numpy as np


def window(y, length=120.0, s=12.0):
    """1 near the end, 0 far from it (y <= 0), smooth to double precision."""
    return 0.5 * np.array([math.erfc(v) for v in (-y - length) / s])


def functional(b, f, m, length=120.0, s=12.0, n=6000):
    """C(b) for h = exp(-i b t): integral up to f minus the regular samples k <= -m."""
    top = math.sqrt(length + 8.0 * s)
    x = (np.arange(n) + 0.5) * top / n                 # t = f - x^2
    wx = 2.0 * window(-x * x) * top / n
    k = np.arange(-int(length + 8.0 * s), 1 - m)
    wk = window(k - f) / np.sqrt(f - k)
    return np.array([np.sum(wx * np.exp(-1j * v * (f - x * x))) - np.sum(wk * np.exp(-1j * v * k)) for v in b])


def table(sigma, m, p, extra, degree, rcond, n_band=300):
    c, w = math.pi / sigma, math.pi / sigma + extra
    b = c + w * np.cos((np.arange(n_band) + 0.5) * math.pi / n_band)
    a = np.exp(-1j * np.outer(b, np.arange(1 - m, p + 1)))
    # the truncated pseudo-inverse, applied factor by factor (its entries are as large as 1 / rcond)
    u, sv, vh = np.linalg.svd(a, full_matrices=False)
    r = int((sv > rcond * sv[0]).sum())
    u, sv, vh = u[:, :r], sv[:r], vh[:r]
    x = np.cos((np.arange(degree + 1) + 0.5) * math.pi / (degree + 1))
    vals = np.array([vh.conj().T @ ((u.conj().T @ functional(b, 0.5 * (t + 1.0), m)) / sv) for t in x])          # (node, tap)
    cheb = np.polynomial.chebyshev.chebvander(x, degree)
    coef = np.linalg.solve(cheb, vals)                                              # Chebyshev
    mono = np.array([np.polynomial.chebyshev.cheb2poly(col) for col in coef.T])     # (tap, power)
    err = 0.0
    for f in (0.0, 0.013, 0.31, 0.5, 0.77, 0.999):
        ws = np.polynomial.polynomial.polyval(2.0 * f - 1.0, mono.T)
        err = max(err, np.abs(a @ ws - functional(b, f, m)).max())
    print("sigma %d: %d + %d weights, degree %d, band +- %.2f, worst error %.1e, largest coefficient %.1f"
          % (sigma, m, p, degree, w, err, np.abs(mono).max()), file=sys.stderr)
    return mono


def emit(name, ctype, mono, fmt):
    taps, n = mono.shape
    print("__device__ const %s %s[%d][%d][2] = {" % (ctype, name, taps, n))
    for row in mono:
        print("    {%s}," % ", ".join("{%s, %s}" % (fmt % v.real, fmt % v.imag) for v in row))
    print("};")


def main():
    print("// Written by gen_end_weights.py: endpoint weights of the back-projection's sample sums,")
    print("// w_j(f) as polynomials in x = 2 f - 1: [weight][power][re, im].  Weight j belongs to the")
    print("// sample floor(u) + 1 - kEndIn + j.")
    print("#pragma once\n\nnamespace cfft {\n")
    print("template <class T>\nstruct EndShape;")
    for t, sig, m, p, d in (("float", 4, 10, 6, 9), ("double", 8, 12, 8, 12)):
        print("template <>\nstruct EndShape<%s> {\n  static constexpr int kSigma = %d, kIn = %d, kOut = %d, kDeg = %d;\n};"
              % (t, sig, m, p, d))
    print()
    emit("kEndWeightsF", "float", table(4, 10, 6, 0.4, 9, 1e-9), "%.9gf")
    emit("kEndWeightsD", "double", table(8, 12, 8, 0.4, 12, 1e-13), "%.17g")
    print("\n}  // namespace cfft")


if __name__ == "__main__":
    main()
