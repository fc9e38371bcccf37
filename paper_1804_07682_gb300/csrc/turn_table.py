"""Generate turn_table.h: cos and sin of 2 pi k / 512 as 64-bit integers
(scale 2^62) and the integer constants of the element-wise probability's
fixed-point evaluation (turns.cuh).

Everything is computed in exact rational arithmetic from the Taylor series and
pi to 60 digits, then rounded to the nearest integer.

Run:  python turn_table.py > turn_table.h
"""
from fractions import Fraction

# pi to 60 digits (textbook value)
PI = Fraction("3.14159265358979323846264338327950288419716939937510582097494")
N = 512


def cos_sin(x):
    """Taylor series to below 1e-30 for |x| <= pi / 4."""
    c, s, term, k = Fraction(0), Fraction(0), Fraction(1), 0
    while abs(term) > Fraction(1, 10 ** 32):
        if k % 2 == 0:
            c += term if k % 4 == 0 else -term
        else:
            s += term if k % 4 == 1 else -term
        k += 1
        term = term * x / k
        term = Fraction(round(term * 10 ** 45), 10 ** 45)
    return c, s


def entry(k):
    """(cos, sin) of 2 pi k / N from the octant of k."""
    q, j = divmod(k + N // 8, N // 4)  # quarter turn q, remainder within +- an eighth
    c, s = cos_sin(2 * PI * (j - N // 8) / N)
    return [(c, s), (-s, c), (-c, -s), (s, -c)][q % 4]


def q(x, bits):
    return round(x * 2 ** bits)


def main():
    print("// Generated by turn_table.py -- do not edit.")
    print("#pragma once")
    print("// 1/pi = GNA_INV_PI_Q65 / 2^65")
    print("#define GNA_INV_PI_Q65 0x%016xull" % q(1 / PI, 65))
    t = 2 * PI
    print("// cos w - 1 = -d^2 (C1 - d^2 (C2 - d^2 C3)), sin w = d (S0 - d^2 (S1 - d^2 S2)), w = 2 pi d;")
    print("// the integers are the coefficients times the power of two in their names")
    for name, x, bits in (("C1_Q58", t ** 2 / 2, 58), ("C2_Q24", t ** 4 / 24, 24), ("C3_Q24", t ** 6 / 720, 24),
                          ("S0_Q60", t, 60), ("S1_Q57", t ** 3 / 6, 57), ("S2_Q24", t ** 5 / 120, 24)):
        print("#define GNA_TURN_%s %dll" % (name, q(x, bits)))
    print("// {cos, sin}(2 pi k / %d) times 2^62" % N)
    print("#define GNA_TURN_TABLE \\")
    rows = []
    for k in range(N):
        c, s = entry(k)
        rows.append("    {%dll, %dll}" % (q(c, 62), q(s, 62)))
    print(", \\\n".join(rows))


if __name__ == "__main__":
    main()
