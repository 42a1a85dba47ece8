"""Write line_table.h: the constants of the compact line solver in lines.cu.

For the interpolation (alpha = 3/10, a/2 = 3/4, b/2 = 1/20) and the derivative (alpha = 9/62,
a = 63/62, b/3 = 17/186): rho with rho / (1 + rho^2) = alpha (1/3 and 0.148309...), its powers 1 to
16, (rho^8 2^FALL)^1, ^2 and ^4, the right-hand side's weights times 1 + rho^2, and the responses of a
segment's rows. Each constant c is held as the pair (h, l) of signed 32-bit words with h 2^32 + l the
integer nearest to c 2^64 (powers) or c 2^62 (weights), and as a binary64 number (the powers of
rho^8 without their power of two). 60-digit decimal arithmetic.
Usage: python gen_line_table.py  (rewrites line_table.h beside this file).
"""
from __future__ import annotations

import decimal
import os

D = decimal.Decimal
decimal.getcontext().prec = 60
LSEG = 8
KINDS = ((D(3) / 10, D(3) / 4, D(1) / 20), (D(9) / 62, D(63) / 62, D(17) / 186))
FALL = (11, 20)        # LINE_FALL_0, LINE_FALL_1 of internal.h


def words(x: D, q: int):
    v = int((x * 2 ** q).to_integral_value(rounding=decimal.ROUND_HALF_EVEN))
    lo = (v + 2 ** 31) % 2 ** 32 - 2 ** 31
    return (v - lo) >> 32, lo


def constants(kind: int):
    """[(value, q, power of two)], in the order of lines.cu's c_line."""
    alpha, wa, wb = KINDS[kind]
    rho = (1 - (1 - 4 * alpha * alpha).sqrt()) / (2 * alpha)
    r2 = rho * rho
    return ([(rho ** k, 64, 0) for k in range(1, 17)] +
            [(rho ** (LSEG * i), 64, FALL[kind] * i) for i in (1, 2, 4)] +
            [(wa * (1 + r2), 62, 0), (wb * (1 + r2), 62, 0), (r2 / (1 - r2), 64, 0)] +
            [(rho ** (k + 1) * (1 - r2 ** (LSEG - k)) / (1 - r2), 64, 0) for k in range(LSEG)])


def render() -> str:
    out = ["// Generated by gen_line_table.py: constants of the compact line solver in lines.cu, per kind\n",
           "// (interpolation, derivative), each as {h, l, binary64}. Do not edit.\n#pragma once\n\n",
           "#define LINE_TABLE_BODY \\\n"]
    for kind in range(2):
        out.append("    { \\\n")
        for v, q, up in constants(kind):
            h, lo = words(v, q + up)
            out.append(f"        {{{h}, {lo if lo > -2 ** 31 else '-2147483647 - 1'}, {float(v).hex()}}}, \\\n")
        out.append("    }" + (", \\\n" if kind == 0 else "\n"))
    return "".join(out)


def main() -> None:
    with open(os.path.join(os.path.dirname(os.path.abspath(__file__)), "line_table.h"), "w") as fh:
        fh.write(render())


if __name__ == "__main__":
    main()
