"""Generate rox_core_tables.h: per-line rational forms of Re w(x + iy) inside the slow zones.

Run: python gen_core_tables.py > rox_core_tables.h   (needs mpmath and scipy; the header is committed)

At fixed y, an even function of x is approximated by N(U)/D(U), U = x^2 / (y^2 + 3/2), D(0) = 1:
  * y >= 0.1: Re w itself, relative error included, with degrees (7,8) falling to (2,3) as y grows;
  * y < 0.1: R = (Re w - e^{y^2 - x^2} cos 2xy) / y, degrees (7,8), with an error that is small
    against Re w / y (the Gaussian part is added separately: no rational function follows it).
The coefficients are those of the rational interpolant at fixed U_j, the points where the best
approximation at the middle of the y interval (y = 0.1 for R) errs by zero (a linearised least
squares fit reweighted towards equal ripple: Sanathanan and Koerner 1963, Lawson 1961). Being
solutions of a linear system analytic in y they are smooth in y, and each is stored as a
polynomial: of degree 7 in t = a log2(y) + b on [-1, 1], for R of degree 3 in y^2.
Re w = Re(exp(-z^2) erfc(-iz)) in 50 digits (mpmath); scipy's wofz only places the U_j.
"""
import hashlib

import mpmath as mp
import numpy as np
from scipy.special import wofz

mp.mp.dps = 50
KAPPA = 1.5
DEG = 7
# y interval, degrees of N and D, largest x of a slow zone there
ROWS = [(0.1, 0.2, 7, 8, 6.5), (0.2, 0.4, 7, 8, 6.5), (0.4, 0.55, 6, 7, 6.5), (0.55, 0.75, 6, 7, 6.5),
        (0.75, 1.0, 6, 7, 22.0), (1.0, 1.5, 5, 6, 7.9), (1.5, 2.0, 5, 6, 8.95), (2.0, 2.5, 4, 5, 9.95),
        (2.5, 3.5, 4, 5, 11.65), (3.5, 5.0, 3, 4, 13.6), (5.0, 7.5, 3, 4, 16.1), (7.5, 11.5, 2, 3, 18.7),
        (11.5, 22.0, 2, 3, 18.8)]
Y_R, X_R, DEG_R = 0.1, 7.0, 3
cheb = np.polynomial.chebyshev


def re_w(x, y):
    return wofz(x + 1j * y).real


def gauss(x, y):
    return np.exp(y * y - x * x) * np.cos(2 * x * y)


def re_w_mp(x, y):
    z = mp.mpc(x, y)
    return (mp.exp(-z * z) * mp.erfc(-1j * z)).real


def r_mp(x, y):
    return (re_w_mp(x, y) - mp.exp(mp.mpf(y) ** 2 - x * x) * mp.cos(2 * x * y)) / y


def nodes(f, weight, y, p, q, X, iters=600):
    """u = x^2 at which the best approximation of type (p, q) to f on [0, X] errs by zero."""
    c = (y * y + KAPPA) * 3
    smax = X * X / (X * X + c)
    s = smax * (1 - np.cos(np.linspace(0, np.pi, 5000))) / 2
    u = s * c / (1 - s)
    x = np.sqrt(u)
    f, weight = f(x) * (u + c), weight(x) / (u + c)
    tn, td = cheb.chebvander(2 * s / smax - 1, p), cheb.chebvander(2 * s / smax - 1, q)
    d, lw, best = np.ones_like(u), np.ones_like(u), None
    for _ in range(iters):
        w = (np.sqrt(lw) * weight / np.abs(d))[:, None]
        z = np.linalg.svd(np.hstack([tn * w, -(f[:, None] * td) * w]), full_matrices=False)[2][-1]
        n, dd = tn @ z[:p + 1], td @ z[p + 1:]
        if dd[0] < 0:
            n, dd = -n, -dd
        e = (n / dd - f) * weight
        m = np.abs(e).max()
        if np.all(dd > 0) and (best is None or m < best[0]):
            best = (m, e.copy())
        lw *= (np.abs(e) / m + 1e-2) ** 0.7
        lw /= lw.mean()
        d = np.abs(dd)
    e = best[1]
    i = np.where(np.sign(e[1:]) != np.sign(e[:-1]))[0]
    uz = u[i] - e[i] * (u[i + 1] - u[i]) / (e[i + 1] - e[i])
    assert len(uz) == p + q + 1, (y, len(uz))
    return uz / (y * y + KAPPA)


def coefficients(f, y, p, q, U):
    n = p + q + 1
    a, b = mp.matrix(n, n), mp.matrix(n, 1)
    for i, Ui in enumerate(U):
        Ui = mp.mpf(float(Ui))
        k = f(mp.sqrt(Ui * (mp.mpf(y) ** 2 + KAPPA)), y)
        for j in range(p + 1):
            a[i, j] = Ui ** j
        for j in range(1, q + 1):
            a[i, p + j] = -k * Ui ** j
        b[i] = k
    s = mp.lu_solve(a, b)
    return [s[i] for i in range(n)]


def table(t, co, p, q):
    """[power of t][slot]: slots 0 .. 7 hold n_0 .., slots 8 .. 15 d_1 .."""
    n = len(t)
    V = mp.matrix(n, n)
    for i, v in enumerate(t):
        for j in range(n):
            V[i, j] = mp.mpf(float(v)) ** j
    out = np.zeros((n, 16))
    for k in range(p + q + 1):
        poly = mp.lu_solve(V, mp.matrix([c[k] for c in co]))
        out[:, k if k <= p else 8 + k - p - 1] = [float(a) for a in poly]
    return out


def row(ya, yb, p, q, X):
    ym = (ya * yb) ** 0.5
    U = nodes(lambda x: re_w(x, ym), lambda x: 1 / re_w(x, ym), ym, p, q, X)
    t = np.cos((2 * np.arange(DEG + 1) + 1) * np.pi / (2 * (DEG + 1)))
    h, c = np.log(yb / ya) / 2, np.log(ya * yb) / 2
    return table(t, [coefficients(re_w_mp, float(np.exp(c + h * v)), p, q, U) for v in t], p, q)


def row_r():
    U = nodes(lambda x: (re_w(x, Y_R) - gauss(x, Y_R)) / Y_R, lambda x: Y_R / re_w(x, Y_R), Y_R, 7, 8, X_R)
    n = DEG_R + 1
    v = Y_R ** 2 * (1 + np.cos((2 * np.arange(n) + 1) * np.pi / (2 * n))) / 2
    return table(v, [coefficients(r_mp, float(np.sqrt(a)), 7, 8, U) for a in v], 7, 8)


def main():
    with open(__file__, "rb") as f:     # checked by the build, which has no mpmath everywhere
        digest = hashlib.sha256(f.read()).hexdigest()
    o = ["/* Generated by gen_core_tables.py -- do not edit. */", "/* generator: sha256 %s */" % digest, "#pragma once",
         "#define ROX_CORE_ROWS %d" % len(ROWS), "#define ROX_CORE_DEG %d" % DEG,
         "#define ROX_CORE_KAPPA %.1ff" % KAPPA,
         "/* lower end of each y interval, and a, b of t = a log2(y) + b */",
         "ROX_TABLE float rox_core_y[%d][3] = {" % len(ROWS)]
    for ya, yb, *_ in ROWS:
        la, lb = np.log2(ya), np.log2(yb)
        o.append("  {%.9ef, %.9ef, %.9ef}," % (ya, 2 / (lb - la), -(la + lb) / (lb - la)))
    o += ["};", "/* [interval][slot][power of t]: n_0 .. in slots 0 .., d_1 .. in slots 8 .. */",
          "ROX_GTABLE ROX_ALIGN16 float rox_core_t[%d][16][%d] = {" % (len(ROWS), DEG + 1)]
    for r in ROWS:
        o.append("{" + ",\n ".join("{" + ", ".join("%.9ef" % v for v in line) + "}" for line in row(*r).T) + "},")
    o.append("};")
    o += ["/* y < 0.1: [slot][power of y^2] */", "#define ROX_CORE_DEG_R %d" % DEG_R,
          "ROX_TABLE float rox_core_r[16][%d] = {" % (DEG_R + 1)]
    o.append(",\n".join("{" + ", ".join("%.9ef" % v for v in col) + "}" for col in row_r().T))
    o.append("};")
    print("\n".join(o))


if __name__ == "__main__":
    main()
