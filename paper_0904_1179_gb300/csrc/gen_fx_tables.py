"""Writes su3_fx_tables.cuh: the tables of the fixed-point logarithm and of the
fixed-point sine and cosine (su3_fx_kp.cuh), rounded to the nearest integer from
40-digit arithmetic.

    python gen_fx_tables.py > su3_fx_tables.cuh
"""
import mpmath

mpmath.mp.dps = 40


def nearest(x):
    return int(mpmath.nint(x))


def literal(v):
    return "%dLL" % v


def main():
    print("// Generated by gen_fx_tables.py.  Do not edit.")
    print("#pragma once\n")
    print("#include <cstdint>\n")
    print("namespace su3dev {\n")
    print("// ln(C / 2048) in units of 2^-57, C = 1024..2048.")
    print("#define SU3_FX_LOG_TABLE \\")
    rows = [literal(nearest(mpmath.log(mpmath.mpf(c) / 2048) * mpmath.mpf(2) ** 57)) for c in range(1024, 2049)]
    print(",\\\n".join("  " + ", ".join(rows[i:i + 5]) for i in range(0, len(rows), 5)))
    print("\n// cos and sin of 2 pi j / 4096 in units of 2^-62, j = 0..512.")
    print("#define SU3_FX_TRIG_TABLE_PAIRS \\")
    rows = []
    for j in range(513):
        x = 2 * mpmath.pi * j / 4096
        rows.append("{%s}" % ", ".join(literal(nearest(f(x) * mpmath.mpf(2) ** 62)) for f in (mpmath.cos, mpmath.sin)))
    print(",\\\n".join("  " + ", ".join(rows[i:i + 2]) for i in range(0, len(rows), 2)))
    print("\n}  // namespace su3dev")


if __name__ == "__main__":
    main()
