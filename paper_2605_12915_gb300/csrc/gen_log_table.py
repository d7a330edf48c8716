"""Generate af_log_table.cuh: the table of the invariants' logarithm (P. T. P. Tang,
"Table-driven implementation of the logarithm function in IEEE floating-point
arithmetic", ACM TOMS 16, 1990; af_reduce.cuh evaluates it).

Point i of 512 is c_i, the double with high word LOG_FIRST + (i << 11) and low word 0,
from 0.70703 to 1.41211; 1 is one of them.  Its entry holds g = 1 / c_i rounded to a
multiple of 2^-13 (so that g m - 1 is exact where c_i is next to 1, whose logarithms are
small) and -log(g) = hi + lo: hi a multiple of 2^-42, so that e * LOG_2_HI + hi (log 2 =
LOG_2_HI + LOG_2_LO split alike) is exact for every exponent e of a double, and lo the
rest as a float.

Run:  python gen_log_table.py  (writes af_log_table.cuh next to this file).
"""
import decimal
import os
import struct
import sys
from fractions import Fraction

POINTS, FIRST = 512, 0x3FE6A000

decimal.getcontext().prec = 60


def dec(x):
    f = Fraction(x)
    return decimal.Decimal(f.numerator) / decimal.Decimal(f.denominator)


def split(x):
    """Decimal x as (multiple of 2^-42, the rest rounded to a float)."""
    hi = float(Fraction(int((x * 2 ** 42).to_integral_value()), 2 ** 42))
    return hi, struct.unpack("f", struct.pack("f", float(x - dec(hi))))[0]


def point(i):
    return struct.unpack(">d", struct.pack(">II", FIRST + (i << 11), 0))[0]


def main(out_path):
    ln2 = split(decimal.Decimal(2).ln())
    lines = [
        "// GENERATED by gen_log_table.py -- do not edit.",
        "// Per point c: g, 1/c to 13 bits, and -log(g) as a multiple of 2^-42 and the rest.",
        "#pragma once",
        "",
        "namespace af {",
        "",
        "constexpr int LOG_POINTS = %d;" % POINTS,
        "constexpr unsigned LOG_FIRST = 0x%xu;  // high word of the first point" % FIRST,
        "constexpr double LOG_2_HI = %s;" % ln2[0].hex(),
        "constexpr float LOG_2_LO = %sf;" % ln2[1].hex(),
        "struct LogEntry {",
        "  double g, hi;",
        "};",
    ]
    g = [round(2 ** 13 / point(i)) / 2 ** 13 for i in range(POINTS)]
    parts = [split(-dec(x).ln()) for x in g]
    lines.append("static __device__ const LogEntry LOG_TABLE[LOG_POINTS] = {")
    lines += ["    {%s, %s}," % (x.hex(), p[0].hex()) for x, p in zip(g, parts)]
    lines += ["};", "static __device__ const float LOG_TABLE_LO[LOG_POINTS] = {"]
    for i in range(0, POINTS, 4):
        lines.append("    " + " ".join("%sf," % p[1].hex() for p in parts[i:i + 4]))
    lines += ["};", "", "}  // namespace af", ""]
    with open(out_path, "w") as f:
        f.write("\n".join(lines))


if __name__ == "__main__":
    here = os.path.dirname(os.path.abspath(__file__))
    main(sys.argv[1] if len(sys.argv) > 1 else os.path.join(here, "af_log_table.cuh"))
