"""Derives the constants of the even part of GELU in mlp_velocity.cu.

    python paper_2509_06040_b200/csrc/gelu_poly_fit.py

GELU(x) = x / 2 + E(x), E(x) = x erf(x / sqrt 2) / 2, which is even.  On |x| <= 1 the kernel evaluates, with y = 2x and
t = y^2,  kappa E(x) = t (R0 + R1 t)  in packed bf16.  The factor kappa is free (it is taken back on the outputs), so of the
two coefficients only the ratio has to suit bf16: for every bf16 R0 in [1, 2) the ratio of the unrounded fit gives R1, and the
pair is kept whose largest error is smallest (weighted least squares with Lawson's reweighting for the fit and for kappa).  Prints the
coefficients, their bf16 bit patterns, kappa and the largest error in exact arithmetic.
"""
import numpy as np
from scipy.special import erf

RANGE = 1.0


def to_bf16(x):
    u = np.asarray(x, dtype=np.float32).reshape(1).view(np.uint32).astype(np.uint64)
    u = (u + 0x7FFF + ((u >> 16) & 1)) & 0xFFFF0000
    return float(u.astype(np.uint32).view(np.float32)[0])


def fit():
    x = np.linspace(1e-3, RANGE, 4000)
    t = 4.0 * x * x
    target = 0.5 * x * erf(x / np.sqrt(2.0))
    basis = np.stack([t, t * t], axis=1)
    weight = np.ones_like(x)
    for _ in range(200):
        coef, *_ = np.linalg.lstsq(basis * weight[:, None], target * weight, rcond=None)
        err = np.abs(basis @ coef - target)
        weight *= 0.5 + err / err.max()
        weight /= weight.max()
    best = None
    for m in range(128, 256):
        r0 = m / 128.0
        r1 = to_bf16(r0 * coef[1] / coef[0])
        poly = t * (r0 + r1 * t)
        kappa = float(np.float32(np.dot(weight * target, weight * poly) / np.dot(weight * target, weight * target)))
        err = np.abs(poly / kappa - target).max()
        if best is None or err < best[0]:
            best = (err, r0, r1, kappa)
    return best


if __name__ == "__main__":
    err, r0, r1, kappa = fit()
    for name, v in (("R0", r0), ("R1", r1)):
        print(f"{name} = {v!r}  bf16 bits 0x{int(np.float32(v).view(np.uint32)) >> 16:04x}")
    print(f"kappa = {kappa!r}; largest |E| error on |x| <= {RANGE:.2f}: {err:.3g}")
