"""Writes int64_tables.h: the fixed-point tables and coefficients of the
integer exp2 and log2 (pr_int64.cuh), from 50-digit arithmetic (mpmath).

    python paper_2312_04830_gb300/csrc/gen_int64_tables.py

exp2: 2^(-j/1024) x 2^63, j = 0..1023, and the Taylor coefficients of 2^-g
for g in [0, 2^-10), the fourth less 0.93 x 2^-10 times the fifth (which
leaves an error of at most 7 % of the fifth term, 2^-63).  log2: for F = 1 +
j/256 the inverse 1/F x 2^64, rounded up by 8 units so that m times it stays
at or above 1 in truncating arithmetic, log2 of that inverse's reciprocal, and
the Taylor coefficients of log2(1 + r).
"""
import os

import mpmath

mpmath.mp.dps = 60
HERE = os.path.dirname(os.path.abspath(__file__))


def fix(v, bits):
    return int(mpmath.nint(mpmath.mpf(v) * mpmath.power(2, bits)))


def array(name, values):
    return "I64_TAB uint64_t %s[%d] = {" % (name, len(values)) + ", ".join("0x%016Xull" % v for v in values) + "};"


def main():
    ln2 = mpmath.log(2)
    lines = ["// Generated by gen_int64_tables.py (60-digit arithmetic); do not edit.", "#pragma once", "#include <stdint.h>", ""]
    lines.append("// 2^(-j/1024), units 2^-63")
    lines.append(array("kI64Exp2", [fix(mpmath.power(2, -mpmath.mpf(j) / 1024), 63) for j in range(1024)]))
    c = [ln2 ** k / mpmath.factorial(k) for k in range(6)]
    c[4] -= mpmath.mpf("0.93") / 1024 * c[5]
    lines.append("// coefficient k = 1..4 of (g 2^10)^k in 2^-g, units 2^-(63 + k)")
    lines.append("constexpr uint64_t kI64ExpC1 = 0x%016Xull, kI64ExpC2 = 0x%016Xull;" % tuple(fix(c[k], 63 + k - 10 * k) for k in (1, 2)))
    lines.append("constexpr uint32_t kI64ExpC3 = 0x%08Xu, kI64ExpC4 = 0x%08Xu;" % tuple(fix(c[k], 63 + k - 10 * k) for k in (3, 4)))
    inv, lg = [0], [0]
    for j in range(1, 256):
        F = 1 + mpmath.mpf(j) / 256
        i = int(mpmath.ceil(mpmath.power(2, 64) / F)) + 8
        inv.append(i)
        lg.append(fix(-mpmath.log(mpmath.mpf(i) / mpmath.power(2, 64), 2), 64))
    lines.append("// 1/F (plus 8 units), units 2^-64, and log2 of its reciprocal, units 2^-64; F = 1 + j/256")
    lines.append(array("kI64InvF", inv))
    lines.append(array("kI64Log2F", lg))
    d = [0] + [1 / (k * ln2) for k in range(1, 8)]
    lines.append("// coefficient k = 1..7 of (r 2^8)^k in log2(1 + r), units 2^-(64 + k) (signs alternate)")
    lines.append("constexpr uint64_t kI64LogC1 = 0x%016Xull, kI64LogC2 = 0x%016Xull, kI64LogC3 = 0x%016Xull, kI64LogC4 = 0x%016Xull;"
                 % tuple(fix(d[k], 64 + k - 8 * k) for k in (1, 2, 3, 4)))
    lines.append("constexpr uint32_t kI64LogC5 = 0x%08Xu, kI64LogC6 = 0x%08Xu, kI64LogC7 = 0x%08Xu;"
                 % tuple(fix(d[k], 64 + k - 8 * k) for k in (5, 6, 7)))
    lines.append("constexpr uint64_t kI64Log2E = 0x%016Xull;   // log2 e, units 2^-63" % fix(1 / ln2, 63))
    lines.append("constexpr uint64_t kI64Ln2 = 0x%016Xull;   // ln 2, units 2^-64" % fix(ln2, 64))
    with open(os.path.join(HERE, "int64_tables.h"), "w") as f:
        f.write("\n".join(lines) + "\n")


if __name__ == "__main__":
    main()
