"""Constants of cell_mass.cuh: the Gaussian mass of a map cell as a polynomial times one exponential.

A cell of half-width t (in units of sigma) whose centre lies at distance z holds the mass

    int_{-t}^{t} phi(z + v) dv = 2 t phi(z) sum_i He_2i(z) u^i / (2i + 1)!,   u = t^2

(Taylor's series of phi under the integral; He_k the probabilists' Hermite polynomials). With
y = z^2 the sum is a polynomial in y whose coefficients are polynomials in u. Powers y^m above the
degree D kept are replaced by the degree-D polynomial nearest to them under the weight exp(-y/2)
that the sum is multiplied by (minimax, by iteratively reweighted least squares). Prints, for the
scaled variable s = y / (2 ln 2) (so that exp(-y/2) = 2^-s), the table c_i = sum_k T[i][k] u^k and
the largest error over the half-widths in use, relative to the mass of the cell at the centre.

    python fit_cell_mass.py
"""
import math

import numpy as np

ORDER = 6  # highest power of u


def hermite_even(i):
    """He_2i as coefficients of y = z^2, lowest first."""
    p = np.polynomial.hermite_e.herme2poly([0] * (2 * i) + [1])
    return p[::2]


def nearest(m, D, ymax=60.0, n=6001):
    """Degree-D coefficients minimising max |exp(-y/2) (y^m - p(y))| on [0, ymax]."""
    y = ymax * (0.5 - 0.5 * np.cos(np.pi * np.arange(n) / (n - 1)))
    w = np.exp(-0.5 * y)
    A = (y[:, None] ** np.arange(D + 1)) * w[:, None]
    b = y ** m * w
    scale = np.abs(A).max(0)
    lam = np.ones(n) / n
    best, best_err = None, np.inf
    for _ in range(4000):  # Lawson's algorithm
        s = np.sqrt(lam)
        c = np.linalg.lstsq(A / scale * s[:, None], b * s, rcond=None)[0] / scale
        e = np.abs(A @ c - b)
        if e.max() < best_err:
            best, best_err = c, e.max()
        lam = lam * e
        lam /= lam.sum()
    return best


def table(D):
    T = np.zeros((D + 1, ORDER + 1))
    near = {m: nearest(m, D) for m in range(D + 1, ORDER + 1)}
    for i in range(ORDER + 1):
        for m, h in enumerate(hermite_even(i)):
            c = h / math.factorial(2 * i + 1)
            if m <= D:
                T[m, i] += c
            else:
                T[:, i] += c * near[m]
    return T


def worst(D, T, tmax):
    """Largest |approximation - mass| over t <= tmax and all z, relative to the mass at z = 0."""
    z = np.linspace(0.0, 8.0, 4001)
    err = 0.0
    for t in np.linspace(tmax / 40, tmax, 40):
        exact = np.array([0.5 * (math.erf((a + t) / math.sqrt(2)) - math.erf((a - t) / math.sqrt(2))) for a in z])
        exact = np.where(z > 4, [0.5 * (math.erfc((a - t) / math.sqrt(2)) - math.erfc((a + t) / math.sqrt(2))) for a in z], exact)
        q = np.zeros_like(z)
        for i in reversed(range(D + 1)):
            q = q * z * z + sum(T[i, k] * t ** (2 * k) for k in range(ORDER + 1))
        got = 2 * t * np.exp(-0.5 * z * z) / math.sqrt(2 * math.pi) * q
        err = max(err, np.abs(got - exact).max() / exact[0])
    return err


if __name__ == "__main__":
    for D, sig in ((3, 1.5), (4, 1.0)):
        T = table(D)
        S = T * (2 * math.log(2)) ** np.arange(D + 1)[:, None]
        for s in (sig, 0.9 * sig, 2.0, 3.0):
            print(f"// D = {D}: sigma = {s:.2f}, half-width sqrt(2)/2 cells: error {worst(D, T, math.sqrt(0.5) / s):.2e} of the peak mass")
        print("{" + ",\n ".join("{" + ", ".join(f"{v:.9e}f" for v in row) + "}" for row in S) + "}")
