"""Prints the coefficients of the polynomial Q in log(1 + f) = f + f^2 Q(f) that the FP32 kernels use
for f in [sqrt(1/2) - 1, sqrt(2) - 1] (log1p_product in lbm_device.cuh): degree 8, minimax for the
relative error of the logarithm, by iteratively reweighted least squares (Lawson's algorithm).

Run:  python tests/golden/make_log1p_polynomial.py
"""
import numpy as np

LO, HI = np.sqrt(0.5) - 1, np.sqrt(2.0) - 1


def fit(degree=8, points=4000, iterations=60):
    """Coefficients by rising power, rounded to FP32, and the relative error before the rounding."""
    a, b = LO - 1e-6, HI + 1e-6
    t = np.cos(np.pi * (np.arange(points) + 0.5) / points)
    f = 0.5 * (a + b) + 0.5 * (b - a) * t
    f = f[np.abs(f) > 1e-6].astype(np.longdouble)
    q = ((np.log1p(f) - f) / f ** 2).astype(float)
    f = f.astype(float)
    weight = np.abs(f ** 2 / np.log1p(f))
    w = np.ones_like(f)
    A = np.vander(f, degree + 1, increasing=True)
    for _ in range(iterations):
        s = weight * np.sqrt(w)
        c = np.linalg.lstsq(A * s[:, None], q * s, rcond=None)[0]
        e = np.abs((A @ c - q) * weight)
        w *= e + 1e-30
        w /= w.mean()
    return c.astype(np.float32), float(e.max())


if __name__ == "__main__":
    c, e = fit()
    print("\n".join(f"f^{k}: {v:.10f}" for k, v in enumerate(c)))
    print(f"relative error {e:.2e}")
