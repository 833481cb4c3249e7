#!/usr/bin/env python3
"""Writes heget_dirtab.h: the breakpoint tables of the integer energy and
azimuth of heget_dir.cuh.

kDirLog[j], j = 0..511, serves mantissas m in [(512 + j)/1024, (513 + j)/1024):
R = ceil(2^30 1024/(512 + j)) (so that m R 2^-30 >= 1) and ln(R 2^-30) in units
of 2^-72, rounded, as three 32-bit words (low first).  kDirAng[j], j = 0..511:
cos and sin of (pi/2) j/512 in units of 2^-63, rounded, at most 2^63 - 1.
Computed with 60-digit decimal arithmetic.  Run from anywhere:
python gen_dirtab.py [output path]"""
import os
from decimal import Decimal, getcontext

getcontext().prec = 60
TABLE = 512


def pi():
    # Machin: pi/4 = 4 atan(1/5) - atan(1/239)
    def atan_inv(x):
        t, s, k, x2 = Decimal(1) / x, Decimal(0), 0, Decimal(x) * x
        while abs(t) > Decimal(10) ** -70:
            s += (t if k % 2 == 0 else -t) / (2 * k + 1)
            t /= x2
            k += 1
        return s
    return 4 * (4 * atan_inv(5) - atan_inv(239))


def cos_sin(a):
    c = s = Decimal(0)
    t, k = Decimal(1), 0
    while abs(t) > Decimal(10) ** -65 or k < 4:
        if k % 2 == 0:
            c += t if k % 4 == 0 else -t
        else:
            s += t if k % 4 == 1 else -t
        k += 1
        t = t * a / k
    return c, s


def main(out=None):
    lines = ["// heget_dirtab.h -- generated by gen_dirtab.py; do not edit.",
             "// Breakpoint tables of heget_dir.cuh: (R, ln R in units of 2^-72, three words) and",
             "// (cos, sin) of (pi/2) j/512 in units of 2^-63.", "#pragma once", "", "namespace heget {", "",
             f"constexpr int kDirTable = {TABLE};",
             f"HEGET_DIR_TABLE uint4 kDirLog[{TABLE}] = {{"]
    for j in range(TABLE):
        R = -((-(1 << 40)) // (TABLE + j))
        v = int(((Decimal(R) / Decimal(1 << 30)).ln() * (1 << 72)).to_integral_value())
        lines.append("    {%s}," % ", ".join(f"0x{w:08x}u" for w in (R & 0xFFFFFFFF, v & 0xFFFFFFFF, v >> 32 & 0xFFFFFFFF, v >> 64)))
    lines += ["};", f"HEGET_DIR_TABLE ulonglong2 kDirAng[{TABLE}] = {{"]
    half_pi = pi() / 2
    for j in range(TABLE):
        c, s = cos_sin(half_pi * j / TABLE)
        w = [min(int((v * (1 << 63)).to_integral_value()), (1 << 63) - 1) for v in (c, s)]
        lines.append(f"    {{0x{w[0]:016x}ull, 0x{w[1]:016x}ull}},")
    ln2 = int((Decimal(2).ln() * (1 << 72)).to_integral_value())
    step = int((half_pi / TABLE * (1 << 71)).to_integral_value())
    lines += ["};", "", "// ln 2 in units of 2^-72 (low, middle, high word); (pi/2)/512 in units of 2^-71",
              "constexpr unsigned kLn2W[3] = {%s};" % ", ".join(f"0x{ln2 >> s & 0xFFFFFFFF:08x}u" for s in (0, 32, 64)),
              f"constexpr unsigned long long kAngStep = 0x{step:016x}ull;", "", "}  // namespace heget", ""]
    out = out or os.path.join(os.path.dirname(os.path.abspath(__file__)), "heget_dirtab.h")
    with open(out, "w") as f:
        f.write("\n".join(lines))


if __name__ == "__main__":
    import sys
    main(sys.argv[1] if len(sys.argv) > 1 else None)
