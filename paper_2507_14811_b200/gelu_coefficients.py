"""Derives the polynomial the fused GELU prologue evaluates (csrc/quantize.cu, gelu2) and prints its
coefficients.  Not used at run time.

erfc(t) = exp(-t^2) g(t) with g the scaled complementary error function.  g is smooth and positive on [0, inf);
with z = (t - c) / (t + c), c = 2.5, the range t in [0, 9.6] (beyond it exp(-t^2) underflows in fp32) maps to
z in [-1, 0.59), and a degree-9 polynomial in z, fitted by least squares on the RELATIVE error at Chebyshev nodes,
reproduces g to 2^-29.  The script also replays the kernel's fp32 operation sequence in numpy over every bf16
input and prints the largest error against h Phi(h) in units of the bound the C header states.
"""
import numpy as np
import scipy.special as sp

C, DEG, T_MAX = 2.5, 9, 9.6
f32 = np.float32


def fit():
    z_max = (T_MAX - C) / (T_MAX + C)
    k = np.arange(6000)
    z = (np.cos(np.pi * (k + 0.5) / 6000) + 1) / 2 * (z_max + 1) - 1
    t = C * (1 + z) / (1 - z)
    g = sp.erfcx(t)
    V = np.polynomial.polynomial.polyvander(z, DEG)
    coef, *_ = np.linalg.lstsq(V / g[:, None], np.ones_like(g), rcond=None)
    return coef


def fma(a, b, c):
    """One rounding: the product of two fp32 numbers is exact in fp64 (its sum with c rounds there first, to 2^-53)."""
    return (a.astype(np.float64) * np.float64(b) + np.float64(c)).astype(f32)


def gelu_f32(h, coef, rcp_ulp):
    """gelu2 of csrc/quantize.cu; rcp_ulp: error of the hardware reciprocal in units of its last place."""
    h = h.astype(f32)
    a = np.minimum(np.abs(h), f32(20.0))
    t = (a * f32(0.70710678118654752440)).astype(f32)
    r = (f32(1.0) / (t + f32(C))).astype(f32)
    r = (r + f32(rcp_ulp) * np.spacing(r)).astype(f32)
    z = ((t - f32(C)).astype(f32) * r).astype(f32)
    g = np.full(h.shape, f32(coef[-1]), f32)
    for c in coef[-2::-1]:
        g = fma(g, z, f32(c))
    s = (t * t).astype(f32)
    neg_e = fma(-t, t, s)                                  # t^2 = s - neg_e exactly
    x = (s * f32(-1.4426950408889634)).astype(f32)
    E = (np.exp2(x.astype(np.float64)).astype(f32) * g).astype(f32)          # subnormal results are kept
    E = fma(E, neg_e, E)
    return fma((a * f32(-0.5)).astype(f32), E, np.maximum(h, f32(0.0)))


if __name__ == "__main__":
    coef = fit()
    print("coefficients, constant term first:")
    print(", ".join("%.9ef" % f32(c) for c in coef))
    h = (np.arange(65536, dtype=np.uint32) << 16).view(np.float32)
    h = h[np.isfinite(h) & (np.abs(h) >= 2.0 ** -100)]
    h64 = h.astype(np.float64)
    with np.errstate(over="ignore", under="ignore"):
        exact = h64 * sp.ndtr(h64)
        bound = (3 * np.minimum(h64 ** 2, 400.0) + 48) * 2.0 ** -24 * np.abs(exact) + np.where(h64 < -13, 2.0 ** -143, 0.0)
        for rcp_ulp in (-1, 0, 1):
            err = np.abs(gelu_f32(h, coef, rcp_ulp).astype(np.float64) - exact)
            near = np.abs(h64) <= 4
            print("every bf16 input, reciprocal off by %d ulp: error at most %.2f of the stated bound; |h| <= 4: 2^%.1f relative"
                  % (rcp_ulp, (err / bound).max(), np.log2((err[near] / np.abs(exact[near])).max())))
