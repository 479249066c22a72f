"""Generates ktrap_tables.h: constants of the trapezoid rule of the K integral
(lb_ktrap.cuh) and of the small-argument series, in fixed point, from mpmath
at 60 digits.

    python3 gen_ktrap.py > ktrap_tables.h

* lb_kt_exp2: 2^(j/2048), j = 0..2047, Q62.
* LB_KT_C1..C3: (2^r - 1)/r = c1 + c2 r + c3 r^2 for 0 <= r < 2^-11, by
  interpolation at the three Chebyshev points of the interval (remainder
  below 2^-58 of 2^r).
* lb_kt_root<m>: 2^(j/m), j = 0..m-1, Q63, for the steps h = ln 2 / m.
* lb_kt32: (e^d - 1 - d, e^-d - 1 + d) at d = k ln2 / m, m = 2, 3, 4 and
  k = 0 .. 63, in single precision, for the FP32 form of the rule.
* LB_KT_G1 / LB_KT_G2: Taylor coefficients in mu^2 of Temme's functions
    Gamma_1(mu) = (1/Gamma(1-mu) - 1/Gamma(1+mu)) / (2 mu),
    Gamma_2(mu) = (1/Gamma(1-mu) + 1/Gamma(1+mu)) / 2
  (N. M. Temme, "On the numerical evaluation of the modified Bessel function
  of the third kind", J. Comput. Phys. 19, 1975), Q62, |mu| <= 1/2.
"""
import mpmath as mp

mp.mp.dps = 60


def q(v, n):
    return int(mp.floor(v * mp.mpf(2) ** n + mp.mpf(1) / 2))


def f32(v):
    return "%sf" % repr(float(mp.nstr(v, 12)))


def table(name, vals, per=4):
    # the kernels copy it to shared memory 16 bytes at a time
    print("alignas(16) LB_IX_TABLE unsigned long long %s[%d] = {" % (name, len(vals)))
    for i in range(0, len(vals), per):
        print("    " + ", ".join("0x%016xull" % v for v in vals[i:i + per]) + ",")
    print("};")


def exp2_poly():
    hw = mp.mpf(2) ** -11
    xs = [hw / 2 * (1 + mp.cos((2 * i + 1) * mp.pi / 6)) for i in range(3)]
    f = [(mp.power(2, r) - 1) / r for r in xs]
    a = mp.lu_solve(mp.matrix([[1, r, r * r] for r in xs]), mp.matrix(f))
    return a[0], a[1], a[2]


def reciprocal_gamma(n):
    """Taylor coefficients of 1/Gamma(1 + z)."""
    return mp.taylor(lambda z: mp.rgamma(1 + z), 0, n)


def main():
    print("// Generated by gen_ktrap.py: do not edit.")
    print("#pragma once")
    print("#if defined(__CUDACC__)")
    print("#define LB_KT32_TABLE static __constant__")
    print("#else")
    print("#define LB_KT32_TABLE static const")
    print("#endif")
    c1, c2, c3 = exp2_poly()
    print("#define LB_KT_C1 0x%016xull   // Q53" % q(c1, 53))
    print("#define LB_KT_C2 0x%08xu       // Q33" % q(c2, 33))
    print("#define LB_KT_C3 0x%08xu       // Q33" % q(c3, 33))
    table("lb_kt_exp2", [q(mp.power(2, mp.mpf(j) / 2048), 62) for j in range(2048)])
    print("// 2^(j/m), Q63")
    for m in (3, 4, 5, 6):
        for j in range(1, m):
            print("#define LB_KT_ROOT%d_%d 0x%016xull" % (m, j, q(mp.power(2, mp.mpf(j) / m), 63)))
    print("// (e^d - 1 - d, e^-d - 1 + d), d = k ln2 / m, m = 2, 3, 4")
    print("LB_KT32_TABLE float lb_kt32[3][64][2] = {")
    for m in (2, 3, 4):
        d = [k * mp.log(2) / m for k in range(64)]
        v = [(mp.expm1(t) - t, mp.expm1(-t) + t) for t in d]
        print("    {" + ", ".join("{%s, %s}" % (f32(p), f32(n)) for p, n in v) + "},")
    print("};")
    c = reciprocal_gamma(19)
    print("// Temme's Gamma_1 and Gamma_2 in mu^2, Q62 (signed)")
    for k in range(9):
        print("#define LB_KT_G1_%d %dll" % (k, q(-c[2 * k + 1], 62)))
    for k in range(9):
        print("#define LB_KT_G2_%d %dll" % (k, q(c[2 * k], 62)))


if __name__ == "__main__":
    main()
