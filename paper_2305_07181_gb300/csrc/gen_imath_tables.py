"""Writes imath_tables.h: the tables of the integer-arithmetic logarithm and
exponential in imath.cuh, computed with 60-digit decimal arithmetic.

  log:  for the 256 intervals of [1, 2), centre c_j = 1 + (j + 1/2)/256:
        r_j = 2^14 / c_j rounded to an integer, and -ln(r_j / 2^14) as an
        integer multiple of 2^-62 (the entry of the exact r_j, not of c_j);
  exp:  2^(j/512), j = 0..511, as an integer multiple of 2^-62;
  ln 2 and ln 2 / 512 as integers of 2^-57 with the rest in units of 2^-89.

    python paper_2305_07181_gb300/csrc/gen_imath_tables.py
"""
from __future__ import annotations

import os
from decimal import ROUND_HALF_EVEN, Decimal, getcontext

getcontext().prec = 60
HERE = os.path.dirname(os.path.abspath(__file__))


def fixed(v: Decimal, bits: int) -> int:
    return int((v * (Decimal(2) ** bits)).to_integral_value(rounding=ROUND_HALF_EVEN))


def render() -> str:
    """The text of imath_tables.h."""
    ln2 = Decimal(2).ln()
    out = ["// Generated by gen_imath_tables.py (60-digit decimal arithmetic); do not edit.", "#pragma once", "",
           "namespace esplit {", "namespace im {", ""]

    def split(name, v):
        hi = fixed(v, 57)
        lo = fixed(v - Decimal(hi) / Decimal(2) ** 57, 89)
        out.append(f"constexpr long long {name}_HI = {hi}LL;  // multiples of 2^-57")
        out.append(f"constexpr int {name}_LO = {lo};  // the rest, multiples of 2^-89")

    split("LN2", ln2)
    split("LN2_512", ln2 / 512)
    out.append(f"constexpr long long LN2_62 = {fixed(ln2, 62)}LL;  // multiples of 2^-62")
    out.append(f"constexpr int INV_LN2_512 = {fixed(512 / ln2, 20)};  // 512 / ln 2, multiples of 2^-20")

    def arr(kind, name, vals, suffix, per):
        out.append(f"IM_TABLE {kind} {name}[{len(vals)}] = {{")
        for i in range(0, len(vals), per):
            out.append("    " + ", ".join(f"{v}{suffix}" for v in vals[i:i + per]) + ",")
        out.append("};")

    r = [int((Decimal(2 ** 14) / (1 + (Decimal(j) + Decimal("0.5")) / 256)).to_integral_value(ROUND_HALF_EVEN))
         for j in range(256)]
    arr("unsigned short", "LOG_R", r, "", 16)
    arr("long long", "LOG_T", [fixed(-(Decimal(v) / 2 ** 14).ln(), 62) for v in r], "LL", 4)
    arr("unsigned long long", "EXP_T", [fixed((Decimal(j) / 512 * ln2).exp(), 62) for j in range(512)], "ULL", 4)
    out += ["", "}  // namespace im", "}  // namespace esplit", ""]
    return "\n".join(out)


def main():
    with open(os.path.join(HERE, "imath_tables.h"), "w") as fh:
        fh.write(render())


if __name__ == "__main__":
    main()
