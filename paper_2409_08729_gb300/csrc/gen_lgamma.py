"""Generates lgamma_table.h: lgamma(t) for 1 <= t < 18 by polynomials.

    python3 gen_lgamma.py > lgamma_table.h

Eight pieces per octave of t (one in the last, [16, 18)).  In a piece with
centre c and half width w, lgamma(c + w s) = sum_k a_k s^k, |s| <= 1, of
degree 12: the interpolation at 13 Chebyshev nodes in 50-digit arithmetic
(the nearest singularity, t = 0, lies at |s| = 17 or more, so the error is
below 1e-18).  Stored as a_k 8^k, for Horner's rule in s/8, in Q57, rounded to
nearest: the error of a step then counts an eighth in the next.
"""
import mpmath as mp

DEG, ROWS = 12, 33


def piece(i):
    e, j = divmod(i, 8)
    w = mp.mpf(2) ** e / 16
    return mp.mpf(2) ** e + (2 * j + 1) * w, w


def coefficients(i):
    c, w = piece(i)
    n = DEG + 1
    s = [mp.cos(mp.pi * (2 * k + 1) / (2 * n)) for k in range(n)]
    A = mp.matrix(n, n)
    b = mp.matrix(n, 1)
    for r in range(n):
        for k in range(n):
            A[r, k] = s[r] ** k
        b[r] = mp.loggamma(c + w * s[r])
    return list(mp.lu_solve(A, b))


def main():
    mp.mp.dps = 50
    print("// Generated by gen_lgamma.py: do not edit.")
    print("#pragma once")
    print("#define LB_LG_DEG %d" % DEG)
    print("#define LB_LG_ROWS %d" % ROWS)
    print("// Q57; [piece][power of s/8, highest first]")
    print("LB_IX_TABLE long long lb_lg[%d][%d] = {" % (ROWS, DEG + 1))
    worst = 0
    for i in range(ROWS):
        a = coefficients(i)
        q = [int(mp.nint(v * 8 ** k * mp.mpf(2) ** 57)) for k, v in enumerate(a)]
        c, w = piece(i)
        for k in range(41):
            s = mp.mpf(k - 20) / 20
            got = sum(mp.mpf(v) * (s / 8) ** p for p, v in enumerate(q)) / 2 ** 57
            worst = max(worst, abs(got - mp.loggamma(c + w * s)))
        print("    {" + ", ".join("%dll" % v for v in reversed(q)) + "},")
    print("};")
    print("// largest error of the rounded polynomials: %s" % mp.nstr(worst, 3))


if __name__ == "__main__":
    main()
