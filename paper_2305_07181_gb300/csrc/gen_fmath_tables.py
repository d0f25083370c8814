"""Writes fmath_tables.h: the tables of the table-driven float64 log and exp
in fmath.cuh (after P. T. P. Tang, "Table-driven implementation of the
exponential function" and "... of the logarithm function in IEEE
floating-point arithmetic", ACM TOMS 15(2), 1989 and 16(4), 1990), computed
here with 50-digit decimal arithmetic:

  log:  c_j = j/128 for j = 91..181 (the grid points of [sqrt(2)/2, sqrt(2)));
        ln(c_j) as a float64 pair hi + lo, and 1/c_j rounded to float64;
  exp:  2^(j/32), j = 0..31, as a float64 pair hi + lo;
  ln 2 split as hi + lo with hi carrying 36 significant bits, so that
  N ln2_hi / 32 and k ln2_hi are exact for |N| < 2^17, |k| < 2^17;
  Taylor coefficients (-1)^(k+1)/k of log1p and 1/k! of expm1.

    python paper_2305_07181_gb300/csrc/gen_fmath_tables.py
"""
from __future__ import annotations

import os
from decimal import Decimal, getcontext

getcontext().prec = 50
HERE = os.path.dirname(os.path.abspath(__file__))


def split(v: Decimal):
    hi = float(v)
    lo = float(v - Decimal(hi))
    return hi, lo


def trunc_bits(v: Decimal, bits: int) -> float:
    """v rounded to a float64 with at most `bits` significant bits."""
    x = float(v)
    import math
    m, e = math.frexp(x)
    scale = 2.0 ** bits
    return math.ldexp(round(m * scale) / scale, e)


def render() -> str:
    """The text of fmath_tables.h."""
    ln2 = Decimal(2).ln()
    ln2_hi = trunc_bits(ln2, 36)
    ln2_lo = float(ln2 - Decimal(ln2_hi))
    l32 = ln2 / 32
    l32_hi = trunc_bits(l32, 36)
    l32_lo = float(l32 - Decimal(l32_hi))
    inv_l32 = float(32 / ln2)
    lines = ["// Generated by gen_fmath_tables.py (50-digit decimal arithmetic); do not edit.", "#pragma once", "",
             "namespace esplit {", "namespace fm {", ""]
    lines.append(f"constexpr double LN2_HI = {ln2_hi!r};")
    lines.append(f"constexpr double LN2_LO = {ln2_lo!r};")
    lines.append(f"constexpr double L32_HI = {l32_hi!r};   // ln2/32, 36 significant bits")
    lines.append(f"constexpr double L32_LO = {l32_lo!r};")
    lines.append(f"constexpr double INV_L32 = {inv_l32!r};  // 32/ln2")
    lines.append("constexpr int LOG_J0 = 91, LOG_J1 = 181;")
    hi, lo, inv = [], [], []
    for j in range(91, 182):
        c = Decimal(j) / 128
        h, l = split(c.ln())
        hi.append(h)
        lo.append(l)
        inv.append(float(Decimal(128) / Decimal(j)))
    def arr(name, vals):
        out = [f"__device__ const double {name}[{len(vals)}] = {{"]
        for i in range(0, len(vals), 3):
            out.append("    " + ", ".join(repr(v) for v in vals[i:i + 3]) + ",")
        out.append("};")
        return out
    lines += arr("LOG_C_HI", hi) + arr("LOG_C_LO", lo) + arr("LOG_INV_C", inv)
    eh, el = [], []
    for j in range(32):
        h, l = split((Decimal(j) / 32 * ln2).exp())
        eh.append(h)
        el.append(l)
    lines += arr("EXP_T_HI", eh) + arr("EXP_T_LO", el)
    # Taylor coefficients
    lines.append("// log1p(r) = r + r^2 (C2 + r (C3 + ... + r C9)),  Ck = (-1)^(k+1)/k (through C12 for")
    lines.append("// the direct series of log1p at |x| < 2^-5)")
    for k in range(2, 13):
        lines.append(f"constexpr double LOG_C{k} = {float(Decimal((-1) ** (k + 1)) / k)!r};")
    lines.append("// expm1(r) = r + r^2 (E2 + r (E3 + ... + r E7)),  Ek = 1/k!")
    f = Decimal(1)
    for k in range(1, 14):
        f *= k
        if k >= 2:
            lines.append(f"constexpr double EXP_E{k} = {float(1 / f)!r};")
    lines += ["", "}  // namespace fm", "}  // namespace esplit", ""]
    return "\n".join(lines)


def main():
    with open(os.path.join(HERE, "fmath_tables.h"), "w") as fh:
        fh.write(render())


if __name__ == "__main__":
    main()
