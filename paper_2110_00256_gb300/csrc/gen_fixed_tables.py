"""Writes fixed_tables.h: the constants of the 64-bit integer logarithm and
exponential in fixed64.cuh, each the nearest integer of a 300-bit evaluation
with mpmath.  Run from this directory:

    python gen_fixed_tables.py > fixed_tables.h
"""
import mpmath as mp

mp.mp.prec = 300


def q(v, bits):
    """The nearest integer to v 2^bits."""
    return int(mp.nint(mp.mpf(v) * mp.mpf(2) ** bits))


def table(name, kind, values, per_line, fmt):
    lines = [f"__device__ const {kind} {name}[{len(values)}] = {{"]
    for i in range(0, len(values), per_line):
        lines.append("    " + ", ".join(fmt(v) for v in values[i:i + per_line]) + ",")
    return lines + ["};"]


def main():
    ln2 = mp.log(2)
    out = ["// Generated by gen_fixed_tables.py (mpmath, 300 bits, nearest integers).", "// Do not edit.", "#pragma once",
           ""]
    k = q(ln2 / 256, 96)
    out += ["// exp: ln2/256 = kExpStep 2^-64 + kExpStepLo 2^-96",
            f"constexpr unsigned long long kExpStep = {hex(k >> 32)}ull;",
            f"constexpr unsigned int kExpStepLo = {hex(k & 0xffffffff)}u;",
            f"constexpr int kExpSteps = {q(256 / ln2, 21)};  // 256/ln2, 2^-21",
            "// log: ln2/2, 2^-63",
            f"constexpr long long kHalfLn2 = {hex(q(ln2 / 2, 63))}ll;",
            ""]
    out.append("// 2^(j/256), 2^-62")
    out += table("kFixExp", "long long", [q(mp.mpf(2) ** (mp.mpf(j) / 256), 62) for j in range(256)], 4,
                 lambda v: hex(v) + "ll")
    r = [q(1 / (1 + (mp.mpf(j) + mp.mpf(1) / 2) / 256), 16) for j in range(256)]
    out.append("// r_j ~ 1/c_j, c_j = 1 + (j + 1/2)/256, 2^-16, and -ln r_j, 2^-63")
    out += table("kFixLogR", "int", r, 8, str)
    out += table("kFixLog", "long long", [q(-mp.log(mp.mpf(v) / 2 ** 16), 63) for v in r], 4, lambda v: hex(v) + "ll")
    # the finer logarithm's: intervals of 1/1024
    r = [q(1 / (1 + (mp.mpf(j) + mp.mpf(1) / 2) / 1024), 16) for j in range(1024)]
    out.append("// the same for c_j = 1 + (j + 1/2)/1024; ln2, 2^-63")
    out.append(f"constexpr long long kLn2 = {hex(q(ln2, 63))}ll;")
    out += table("kFineLogR", "unsigned short", r, 12, str)
    out += table("kFineLog", "long long", [q(-mp.log(mp.mpf(v) / 2 ** 16), 63) for v in r], 4, lambda v: hex(v) + "ll")
    print("\n".join(out))


if __name__ == "__main__":
    main()
