"""Generates the polynomial behind the CUDA path's GELU (csrc/pic_gelu.cuh).

GELU(z) = z Phi(z), Phi(z) = (1 + erf(z / sqrt 2)) / 2.  With a = |z|,

    GELU(z) = max(z, 0) - a Phi(-a),   Phi(-a) ~= 2^q(a),

q of degree 6 on 0 <= a <= Z, Z = 5.8: log2 Phi(-a) is close to a parabola,
so a low degree does.  Beyond Z the subtracted part, below 2e-8, is to vanish
exactly: a is clamped at Z, and the kernels subtract EPS, a little more than
2^q(Z), from the power and clamp the difference at zero.  An error d in q
is an error a Phi(-a) ln 2 d of the GELU, so q is fitted to log2 Phi(-a)
with that weight; Lawson's reweighting raises the weight of the points where
the error is largest, turning the least-squares fit into a minimax one.  It
runs in the scaled variable a / Z on Chebyshev nodes of [0, Z]; the
coefficients are then rescaled for -a, the variable that the kernels keep
(so that the last step is a multiply-add).  Per value the kernels take two
minima or maxima, 6 multiply-adds by Horner's rule, one 2^x (ex2.approx, on
the special-function unit), a saturating subtraction and the last
multiply-add.  The maximum GELU error over the real line with the fp32
evaluation order of the kernels (measured below on a grid of 1.2 M points of
[-12, 12], the power correctly rounded) is printed into the header; most of
it is the rounding of the result itself.

Run:  python -m paper_2609_09020_gb300.gen_gelu  (prints the header)
"""
from __future__ import annotations

import numpy as np
from scipy.special import erf, erfc

Z = 5.8
DEG = 6
PASSES = 200


def fit():
    """Coefficients of q as a polynomial in -a, lowest degree first, and EPS."""
    n = 12000
    a = 0.5 * Z * (1 - np.cos(np.pi * (np.arange(n) + 0.5) / n))
    phi = 0.5 * erfc(a / np.sqrt(2))
    f = np.log2(phi)
    w = a * phi * np.log(2)
    v = (a[:, None] / Z) ** np.arange(DEG + 1)
    lw = np.ones_like(a)
    best = None
    for _ in range(PASSES):
        wt = w * lw
        c, *_ = np.linalg.lstsq(v * wt[:, None], f * wt, rcond=None)
        e = np.abs((v @ c - f) * w)
        if best is None or e.max() < best[0]:
            best = (e.max(), c.copy())
        lw *= np.sqrt(e / e.max() + 1e-3)
        lw /= lw.max()
    c = best[1] * (-1.0 / Z) ** np.arange(DEG + 1)
    return c, float(2.0 ** np.polyval(c[::-1], -Z) * (1 + 1e-3))


def _fma32(a, b, c):
    """fp32 fused multiply-add: the product of two fp32 values is exact in
    fp64, so one rounding of the fp64 sum to fp32 stands in for the FMA's."""
    return (a.astype(np.float64) * b + np.asarray(c, np.float64)).astype(np.float32)


def gelu_fp32(z: np.ndarray, coeffs) -> np.ndarray:
    """fp32 emulation of the CUDA evaluation order (the scalar and the pair
    form round identically: every step is one correctly rounded fp32
    operation; the power is taken correctly rounded here, within two ulps of
    the kernels' ex2.approx)."""
    c, eps = coeffs
    f32 = np.float32
    z = z.astype(f32)
    na = np.maximum(-np.abs(z), f32(-Z))
    q = np.full_like(z, f32(c[-1]))
    for k in c[-2::-1]:
        q = _fma32(q, na, float(f32(k)))
    e = np.exp2(q.astype(np.float64)).astype(f32)
    e = np.clip((e - f32(eps)).astype(f32), 0, 1)
    return _fma32(na, e.astype(np.float64), np.maximum(z, f32(0)))


def min_denominator(coeffs) -> float:
    """The smallest value that the evaluation divides by: it has no division."""
    return 1.0


def max_error(coeffs) -> float:
    z = np.linspace(-12, 12, 1_200_001)
    ref = 0.5 * z * (1 + erf(z / np.sqrt(2)))
    return float(np.max(np.abs(gelu_fp32(z, coeffs).astype(np.float64) - ref)))


def header(coeffs) -> str:
    c, eps = coeffs
    lines = ["// Generated by paper_2609_09020_gb300/gen_gelu.py -- do not edit.",
             f"// Phi(-a) ~= 2^q(-a) on 0 <= a <= {Z}; max |GELU error| in fp32 ~ {max_error(coeffs):.1e}.",
             "#pragma once", "", "namespace pic {", "",
             f"constexpr float kGeluZ = {float(np.float32(Z))!r}f;",
             f"constexpr float kGeluEps = {float(np.float32(eps))!r}f;  // just above 2^q(-Z)",
             f"constexpr int kGeluDeg = {DEG};",
             "",
             "// Coefficients of q, highest degree first (Horner order).",
             "__host__ __device__ constexpr float gelu_c(int i) {",
             "  constexpr float c[] = {"]
    lines += [f"      {float(np.float32(k))!r}f," for k in c[::-1]]
    lines += ["  };", "  return c[i];", "}", "", "}  // namespace pic", ""]
    return "\n".join(lines)


if __name__ == "__main__":
    print(header(fit()))
