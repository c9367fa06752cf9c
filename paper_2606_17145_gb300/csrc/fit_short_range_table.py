"""Writes short_range_table.inc: the piecewise polynomials used by the FP64
walk for the short-range factor of the TreePM split,

    f(u) = erfc(u) + (2 u / sqrt(pi)) exp(-u^2),   u = r / (2 r_s),

on u in [0, 2.25] (the cut rcut = 4.5 r_s).  Interval i is [i, i + 1) / 64; its
entry holds the centre and the coefficients of the degree-6 polynomial in the
offset from the centre that interpolates f at the interval's Chebyshev nodes
(evaluated with 40 digits by mpmath).  The interpolation error is below 1e-17.

Run: python fit_short_range_table.py  (needs mpmath).
"""
import os

PER_UNIT = 64
N = 144  # 2.25 * PER_UNIT
DEG = 6


def entries():
    import mpmath as mp
    mp.mp.dps = 40

    def f(u):
        return mp.erfc(u) + 2 * u / mp.sqrt(mp.pi) * mp.exp(-u * u)

    half = mp.mpf(1) / (2 * PER_UNIT)
    nodes = [half * mp.cos(mp.pi * (2 * k + 1) / (2 * (DEG + 1))) for k in range(DEG + 1)]
    V = mp.matrix(DEG + 1, DEG + 1)
    for i, x in enumerate(nodes):
        for j in range(DEG + 1):
            V[i, j] = x ** j
    out = []
    for i in range(N):
        c = (mp.mpf(i) + mp.mpf(1) / 2) / PER_UNIT
        p = mp.lu_solve(V, mp.matrix([f(c + x) for x in nodes]))
        out.append([float(c)] + [float(v) for v in p])
    return out


def main():
    lines = ["// Generated by fit_short_range_table.py -- do not edit.",
             "// Interval i of width 1 / OG_SR_TABLE_PER_UNIT: centre, then c_0 .. c_6 of",
             "// f(u) = erfc(u) + (2 u / sqrt(pi)) exp(-u^2) = sum_k c_k (u - centre)^k.",
             f"#define OG_SR_TABLE_N {N}",
             f"#define OG_SR_TABLE_PER_UNIT {PER_UNIT}",
             f"static __device__ const double __align__(16) og_sr_table[{8} * OG_SR_TABLE_N] = {{"]
    lines += ["    " + ", ".join(repr(v) for v in e) + "," for e in entries()]
    lines += ["};", ""]
    with open(os.path.join(os.path.dirname(os.path.abspath(__file__)), "short_range_table.inc"), "w") as fh:
        fh.write("\n".join(lines))


if __name__ == "__main__":
    main()
