"""Write log_table.cuh, the table of the FP64 logarithm of the lubrication term.

The method is the table-driven logarithm of P. T. P. Tang, "Table-driven
implementation of the logarithm function in IEEE floating-point arithmetic",
ACM Trans. Math. Softw. 16(4), 1990: x = 2^k m, m in [1, 2), F_j = 1 + j/128
the table point nearest m, and ln x = k ln 2 + ln F_j + ln(1 + (m - F_j)/F_j).
Per j = 0..128 the table holds F_j, 1/F_j rounded to double, and ln F_j as an
unevaluated sum hi + lo with hi a multiple of 2^-42; ln 2 is split the same
way, so that k ln2_hi + hi is exact for |k| < 2^11.  The values come from
mpmath at 60 significant digits.

The second table serves the integer logarithm of the pair kernel (fx.cuh): for
m in [1, 2) and j the leading seven bits of its fraction, C_j = 2^16/(1 + (j +
1/2)/128) rounded to an integer and -ln(C_j/2^16) in units of 2^-58, so that
ln m = ln(1 + u) - ln(C_j/2^16) with u = m C_j/2^16 - 1, |u| < 2^-7.9.

    python gen_log_table.py    # rewrites log_table.cuh beside this file
"""
import os

import mpmath as mp

mp.mp.dps = 60
GRID = mp.mpf(2) ** -42


def split(v):
    hi = mp.nint(v / GRID) * GRID
    return float(hi), float(v - hi)


def main():
    rows = []
    for j in range(129):
        F = mp.mpf(1) + mp.mpf(j) / 128
        hi, lo = split(mp.log(F))
        assert float(F) == 1.0 + j / 128.0
        rows.append((float(F), float(mp.mpf(1) / F), hi, lo))
    l2hi, l2lo = split(mp.log(2))
    out = ["// log_table.cuh -- generated by gen_log_table.py; do not edit.",
           "// Per j = 0..128: F_j = 1 + j/128, 1/F_j, ln F_j = hi + lo (hi a multiple of 2^-42).",
           "#pragma once",
           f"#define DPS_LN2_HI {l2hi.hex()}",
           f"#define DPS_LN2_LO {l2lo.hex()}",
           "#define DPS_LOG_TABLE_ROWS \\"]
    for k, (F, inv, hi, lo) in enumerate(rows):
        sep = "," if k < 128 else ""
        out.append(f"    {{{F.hex()}, {inv.hex()}, {hi.hex()}, {lo.hex()}}}{sep} \\")
    out.append("")
    out.append("// Per j = 0..127: C_j = 2^16/(1 + (j + 1/2)/128) rounded, -ln(C_j/2^16) in units of 2^-58.")
    out.append(f"#define DPS_FX_LN2_Q58 {int(mp.nint(mp.log(2) * mp.mpf(2) ** 58))}LL")
    out.append("#define DPS_FX_LOG_ROWS \\")
    for j in range(128):
        C = int(mp.nint(mp.mpf(2) ** 16 / (1 + (mp.mpf(j) + mp.mpf("0.5")) / 128)))
        T = int(mp.nint(-mp.log(mp.mpf(C) / 2 ** 16) * mp.mpf(2) ** 58))
        out.append(f"    {{{C}LL, {T}LL}}{',' if j < 127 else ''} \\")
    out.append("")
    path = os.path.join(os.path.dirname(os.path.abspath(__file__)), "log_table.cuh")
    with open(path, "w") as f:
        f.write("\n".join(out) + "\n")


if __name__ == "__main__":
    main()
