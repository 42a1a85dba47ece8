"""Write fix_table.h: the constants of the integer exponential and logarithm in fix64.cuh.

In 60-digit decimal arithmetic, each rounded to the nearest integer:
  * 2^(j/256) 2^62 for j = 0..255 (the exponential's table);
  * ln2/256 2^72 (its reduction step) and 256/ln2 2^19 (the reduction index comes from a 32-bit
    product with it; rounded down);
  * inv_j = 2^64 / c_j, c_j = 1 + (j + 1/2) / 128, j = 0..127, and -ln(inv_j 2^-64) 2^58 (the
    logarithm's table); ln2 2^58.
Usage: python gen_fix_table.py  (rewrites fix_table.h beside this file).
"""
from __future__ import annotations

import decimal
import os

D = decimal.Decimal
decimal.getcontext().prec = 60
LN2 = D(2).ln()


def nearest(x: D) -> int:
    return int(x.to_integral_value(rounding=decimal.ROUND_HALF_EVEN))


def tables():
    """(exp_table, C72, K27, log_rows, LN2_58); log_rows[j] = (inv_j, -ln(inv_j 2^-64) 2^58)."""
    exp_table = [nearest((D(j) / 256 * LN2).exp() * 2 ** 62) for j in range(256)]
    rows = []
    for j in range(128):
        inv = nearest(2 ** 64 / (1 + (D(j) + D("0.5")) / 128))
        rows.append((inv, nearest(-(D(inv) / 2 ** 64).ln() * 2 ** 58)))
    return exp_table, nearest(LN2 / 256 * 2 ** 72), int(256 / LN2 * 2 ** 19), rows, nearest(LN2 * 2 ** 58)


def render() -> str:
    table, c72, k19, rows, ln2 = tables()
    out = ["// Generated by gen_fix_table.py: constants of the integer exponential and logarithm in\n",
           "// fix64.cuh. Do not edit.\n#pragma once\n\n",
           f"#define FIX_EXP_C72 0x{c72:016x}ull   // ln2/256 in units of 2^-72\n",
           f"#define FIX_EXP_K19 {k19}            // 256/ln2 in units of 2^-19, rounded down\n",
           f"#define FIX_LN2_58 0x{ln2:016x}ull    // ln2 in units of 2^-58\n",
           "// 2^(j/256), j = 0..255, in units of 2^-62\n",
           "#define FIX_EXP_BODY \\\n"]
    for j in range(0, 256, 4):
        out.append("    " + ", ".join(f"0x{t:016x}ull" for t in table[j:j + 4])
                   + (", \\\n" if j < 252 else "\n"))
    out.append("// per j = 0..127: inv_j = 1 / (1 + (j + 1/2) / 128) in units of 2^-64, -ln(inv_j) in units\n"
               "// of 2^-58\n")
    out.append("#define FIX_LOG_BODY \\\n")
    for j, (inv, t) in enumerate(rows):
        out.append(f"    {{0x{inv:016x}ull, 0x{t:016x}ull}}" + (", \\\n" if j < 127 else "\n"))
    return "".join(out)


def main() -> None:
    with open(os.path.join(os.path.dirname(os.path.abspath(__file__)), "fix_table.h"), "w") as fh:
        fh.write(render())


if __name__ == "__main__":
    main()
