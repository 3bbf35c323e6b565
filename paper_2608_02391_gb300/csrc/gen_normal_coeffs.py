"""Build step: fit the table of the GPU's fast standard-normal quantile.

The GPU maps a Philox word to x = 2u - 1 (exact in fp32), then to
    eps = sqrt(2) erfinv(x) = x * R(L),   L = log2(1 - x^2)  (L <= 0),
with R a parabola in L on each of the segments |L + i / S| <= 1 / (2 S), S = 8, whose
coefficients (a, b, c), R = (c L + b) L + a, are read from a table at
i = round(-S L) = 0 .. S |L|_max.  x lies on the odd lattice m 2^-22 - 1 (m odd,
|x| <= 1 - 2^-22), so L >= log2(2^-21 - 2^-44) > -21 - 2^-22.

R is smooth in L (its cubic term is below 1.1e-3 per unit of L), so the parabolas are within
6e-8 of it, relative, and their rounding dominates: evaluated in fp32 the max relative
error over all 2^22 words is 1.9e-7 and the root mean square 5.1e-8, where one polynomial
of degree 9 for L >= -10 and one of degree 8 in sqrt(-L) for the tail reached 3.2e-7 and
1.3e-7.  S = 6 still gives 2.6e-7 and 8.0e-8, S = 12 1.6e-7 and 4.5e-8.

Each segment is fitted by Chebyshev-node weighted least squares with Lawson reweighting
toward the minimax relative error, against scipy.special's quantile in fp64; after b and c
are rounded to fp32, a is re-centred on the remaining error.

Run: python gen_normal_coeffs.py  -> rewrites normal_coeffs.h beside this script.
"""
import os

import numpy as np
from scipy.special import erfinv, ndtri

S = 8             # segments per unit of L
L_MIN = -21.0625  # below every L the transform can see, with room for lg2.approx's error


def ratio_of_L(L):
    """R(L) = sqrt(2) erfinv(x) / x with x = sqrt(1 - 2^L)."""
    x = np.sqrt(-np.expm1(L * np.log(2.0)))
    with np.errstate(divide="ignore"):
        one_minus_x = -np.expm1(0.5 * np.log1p(-np.exp2(L)))  # accurate where x is close to 1
    eps = np.where(L < -1.0, -ndtri(np.minimum(one_minus_x, 1.0) / 2.0), np.sqrt(2.0) * erfinv(x))
    return np.where(x > 1e-12, eps / np.where(x > 1e-12, x, 1.0), np.sqrt(np.pi / 2))


def fit_segment(i, nodes=300, iters=25):
    lo, hi = -(i + 0.5) / S, min(-(i - 0.5) / S, 0.0)
    mid = (lo + hi) / 2
    z = lo + (np.cos(np.linspace(0, np.pi, nodes)) + 1) * (hi - lo) / 2
    y = ratio_of_L(z)
    w = 1.0 / np.abs(y)
    A = np.vander((z - mid) * S, 3, increasing=True)
    for _ in range(iters):
        c, *_ = np.linalg.lstsq(A * w[:, None], y * w, rcond=None)
        err = (A @ c - y) / y
        w = w * np.sqrt(np.abs(err) / np.abs(err).max()) + 1e-300
        w /= w.max()
    p = np.poly1d(c[::-1])(np.poly1d([S, -mid * S]))  # in powers of L
    b, cc = np.float32(p[1]), np.float32(p[2])
    rest = y - (float(cc) * z + float(b)) * z
    return np.float32((rest.max() + rest.min()) / 2), b, cc


def fma(a, b, c):
    return (a.astype(np.float64) * b + c).astype(np.float32)  # one rounding


def main():
    n = int(round(-S * L_MIN)) + 1
    table = np.array([fit_segment(i) for i in range(n)], np.float32)
    t = np.arange(1, 1 << 22, 2, dtype=np.float64) * 2.0**-22  # 1 - |x| of every word
    x = 1.0 - t
    eps = -ndtri(t / 2)
    L = np.log2(fma(-x, x, 1.0).astype(np.float64)).astype(np.float32)
    i = (fma(L, -float(S), 2.0**23).view(np.uint32) - 0x4B000000).astype(np.int64)
    assert i.min() == 0 and i.max() < n
    r = fma(fma(table[i, 2], L, table[i, 1]), L, table[i, 0])
    rel = (x * r).astype(np.float32) / eps - 1.0
    worst, rms = np.abs(rel).max(), np.sqrt(np.mean(rel**2))
    here = os.path.dirname(os.path.abspath(__file__))
    with open(os.path.join(here, "normal_coeffs.h"), "w") as fh:
        fh.write("// Generated by gen_normal_coeffs.py -- do not edit.\n")
        fh.write("// Parabolas of the fast standard-normal quantile eps = x * R(L), L = log2(1 - x^2):\n")
        fh.write("// R = (c L + b) L + a with (a, b, c, 0) the entry round(-SEGMENTS L).\n")
        fh.write(f"// Relative error of eps over all words (simulated): max {worst:.2e}, rms {rms:.2e}.\n#pragma once\n\n")
        fh.write(f"#define COPES_NORMAL_SEGMENTS {S}  // per unit of L\n")
        fh.write(f"#define COPES_NORMAL_ENTRIES {n}\n")
        fh.write("#define COPES_NORMAL_TABLE { \\\n")
        for a, b, c in table:
            fh.write("  {" + ", ".join(f"{v.item():.9e}f" for v in (a, b, c)) + ", 0.0f}, \\\n")
        fh.write("}\n")
    print(f"{n} entries, max rel {worst:.3e}, rms {rms:.3e}")


if __name__ == "__main__":
    main()
