"""Writes haar_tables.h: the tables of the fixed-point Haar sampler (haar_fixed.h).
Run once, from this directory:

    python gen_haar_tables.py > haar_tables.h

Values are computed at 60 significant digits (sympy) and rounded to the nearest integer:
  cos, sin(2 pi k / 512) in units of 2^-60 as 30-bit halves (h, l: h 2^30 + l), k = 0..511
  r_j = 1 / (3/4 + j/512) in units of 2^-63 and ln r_j (of the rounded r_j) in units of
  2^-62, j = 0..384 (r_128 = 1)
"""
import sympy as sp

DIG = 60


def fix(x, bits):
    return int(sp.floor(x * sp.Integer(2) ** bits + sp.Rational(1, 2)))


def main():
    out = ["// haar_tables.h -- generated by gen_haar_tables.py (do not edit): tables of the",
           "// fixed-point Haar sampler.",
           "#pragma once", "#include <cstdint>", ""]
    out.append("// cos, sin(2 pi k / 512) in units of 2^-60 as 30-bit halves, k = 0..511")
    out.append("FP_TABLE int32_t kCosSin[2048] = {")
    for k in range(512):
        a = sp.pi * sp.Rational(k, 256)
        c, s = fix(sp.cos(a).evalf(DIG), 60), fix(sp.sin(a).evalf(DIG), 60)
        out.append(f"    {c >> 30}, {c & 0x3FFFFFFF}, {s >> 30}, {s & 0x3FFFFFFF},")
    out.append("};")
    out.append("")
    out.append("// r_j = 1 / (3/4 + j/512) in units of 2^-63, ln r_j in units of 2^-62, j = 0..384")
    out.append("FP_TABLE int64_t kRecLog[770] = {")
    for j in range(385):
        r = fix((1 / (sp.Rational(3, 4) + sp.Rational(j, 512))).evalf(DIG), 63)
        t = fix(sp.log(sp.Rational(r, 2 ** 63)).evalf(DIG), 62)
        out.append(f"    (int64_t){r}ULL, {t}LL,")
    out.append("};")
    print("\n".join(out))


if __name__ == "__main__":
    main()
