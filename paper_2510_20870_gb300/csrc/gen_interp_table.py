"""Generate rox_interp_table.h: from the values of a smooth function at the 32 Chebyshev points
of a span to its 256 grid points.

Run: python gen_interp_table.py > rox_interp_table.h  (build() does, into the build folder)

On a uniform grid a span's points are x_j = (2j - 255)/255, j = 0..255, on [-1, 1] and the
Chebyshev points (first kind) xi_k = cos((2k + 1) pi / 64), k = 0..31. The table holds the
Lagrange cardinal functions l_k(x_j) of those points, from the barycentric formula (Berrut and
Trefethen, SIAM Review 46 (2004) 501-517, weights (-1)^k sin((2k + 1) pi / 64)), in double
precision, stored as [sub-span m][k][lane] for the point j = 32 m + lane.
"""
import math

SPAN, N = 256, 32


def main():
    xi = [math.cos((2 * k + 1) * math.pi / (2 * N)) for k in range(N)]
    wt = [(-1) ** k * math.sin((2 * k + 1) * math.pi / (2 * N)) for k in range(N)]
    rows = []
    for j in range(SPAN):
        x = (2.0 * j - (SPAN - 1)) / (SPAN - 1)
        t = [w / (x - c) for w, c in zip(wt, xi)]      # no grid point is a Chebyshev point
        s = math.fsum(t)
        rows.append([v / s for v in t])
    out = ["/* Generated by gen_interp_table.py -- do not edit. */", "#pragma once",
           "/* Chebyshev points of a span on [-1, 1] and their barycentric weights */",
           "static __constant__ const float rox_cheb_x[%d] = {%s};" % (N, ", ".join("%.9ef" % v for v in xi)),
           "static __constant__ const float rox_cheb_w[%d] = {%s};" % (N, ", ".join("%.9ef" % v for v in wt)),
           "/* l_k(x_j) at [m][k][lane], j = 32 m + lane */",
           "static __device__ const float rox_interp[%d][%d][32] = {" % (SPAN // 32, N)]
    for m in range(SPAN // 32):
        out.append("{" + ",\n".join("{" + ",".join("%.8ef" % rows[32 * m + i][k] for i in range(32)) + "}"
                                   for k in range(N)) + "},")
    out.append("};")
    print("\n".join(out))


if __name__ == "__main__":
    main()
