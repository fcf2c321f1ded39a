"""Writes noise_fx_tables.cuh: the tables of the fixed-point Box-Muller
functions (noise_fx.cuh), computed from their definitions with the 50-digit
decimal arithmetic of bm_tables.py and rounded once.

  LN_TAB[i]  = (R_i, ln(R_i / 512) 2^57), i the 7 bits after the leading one of
               a significand m in [1, 2): c = the middle of its cell, halved for
               i >= FOLD (m >= sqrt 2), R_i = the integer nearest to 512 / c;
               i = 127 (the cell below 1 after halving) has R = 512 exactly
  LN2        = ln 2 in units of 2^-57
  SC_TAB[j]  = sin(pi j / 64), cos(pi j / 64) as fixed-point numbers (l, h), j = 0 .. 128

Run from this directory: python noise_fx_tables.py > noise_fx_tables.cuh
"""
from decimal import Decimal

from bm_tables import PI, sin_cos

FOLD = 53  # 1 + 53 / 128 < sqrt 2 < 1 + 54 / 128


def nearest(x):
    return int(x.to_integral_value())


def reciprocal(i):
    if i == 127:
        return 512
    c = (Decimal(257 + 2 * i) / 256) / (2 if i >= FOLD else 1)
    return nearest(512 / c)


def split(v):
    h = (v + (1 << 29)) >> 30
    return h, v - (h << 30)


def main():
    out = ["// noise_fx_tables.cuh -- generated by noise_fx_tables.py; do not edit.",
           "// Tables of the fixed-point Box-Muller ln and sincospi (noise_fx.cuh).", "#pragma once",
           "#include <cuda_runtime.h>", "", "namespace clgc {", "",
           "const int NFX_LN_FOLD = %d;" % FOLD,
           "const long long NFX_LN2 = %dll;  // ln 2 2^57" % nearest(Decimal(2).ln() * 2 ** 57), "",
           "// (R, ln(R / 512) 2^57)", "__device__ const longlong2 NFX_LN_TAB[128] = {"]
    for i in range(128):
        r = reciprocal(i)
        out.append("    {%dll, %dll}," % (r, nearest((Decimal(r) / 512).ln() * 2 ** 57)))
    out += ["};", "", "// (sin l, sin h, cos l, cos h) of pi j / 64, x = (h 2^30 + l) 2^-60",
            "__device__ const int4 NFX_SC_TAB[129] = {"]
    for j in range(129):
        s, c = sin_cos(PI * j / 64)
        hs, ls = split(nearest(s * 2 ** 60))
        hc, lc = split(nearest(c * 2 ** 60))
        out.append("    {%d, %d, %d, %d}," % (ls, hs, lc, hc))
    out += ["};", ""]
    for name, v in (("NFX_PI_4", PI / 4), ("NFX_RSQRT3", 1 / Decimal(3).sqrt())):
        h, l = split(nearest(v * 2 ** 60))
        out.append("const int %s_H = %d, %s_L = %d;" % (name, h, name, l))
    out += ["", "}  // namespace clgc"]
    print("\n".join(out))


if __name__ == "__main__":
    main()
