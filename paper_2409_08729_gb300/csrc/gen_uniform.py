"""Generates uniform_tables.h: the Debye polynomials of the uniform expansion in
64-bit fixed point (lb_uniform.cuh), from the exact rationals of gen_debye.py.

    python3 gen_uniform.py > uniform_tables.h

P_k(p) = sum_i c_i p^i has alternating signs, so P_k = E(p^2) - p O(p^2) with
E, O of positive coefficients.  With y = p^2/2, g = p/2 and 8/r as variables
(Q64 integers below 2^63), the entries are

    E: |c_2i| 2^i / 8^k,   O: |c_(2i+1)| 2^(i+1) / 8^k      (Q56)

as pairs (E_i, O_i), i = 0 .. k // 2, for k = 1 .. 13 in turn.  The second
table holds Q_k = k P_k + 2 p P_k', for the x-derivative: the same entries
times k + 2 (2i) and k + 2 (2i + 1), in Q50.
"""
from gen_debye import debye_polys


def main():
    u = debye_polys(13)
    rows, drows, offs = [], [], [0, 0]
    for k in range(1, 14):
        c = [u[k].get(k + 2 * i, 0) for i in range(k + 1)]
        assert all((a > 0) == (i % 2 == 0) for i, a in enumerate(c))
        for i in range(k // 2 + 1):
            e = abs(c[2 * i]) * 2 ** i / 8 ** k
            o = abs(c[2 * i + 1]) * 2 ** (i + 1) / 8 ** k if 2 * i + 1 <= k else 0
            rows.append(tuple(int(round(a * 2 ** 56)) for a in (e, o)))
            drows.append(tuple(int(round(a * 2 ** 50)) for a in ((k + 4 * i) * e, (k + 4 * i + 2) * o)))
        offs.append(len(rows))
    print("// Generated by gen_uniform.py: do not edit.")
    print("#pragma once")
    print("#if defined(__CUDACC__)")
    print("#define LB_UNI_TABLE static __constant__")
    print("#else")
    print("#define LB_UNI_TABLE static const")
    print("#endif")
    print("LB_UNI_TABLE int lb_uni_off[15] = {%s};" % ", ".join(map(str, offs)))
    for name, t in (("lb_uni", rows), ("lb_uniq", drows)):
        print("LB_UNI_TABLE unsigned long long %s[%d][2] = {" % (name, len(t)))
        for e, o in t:
            print("    {0x%016xull, 0x%016xull}," % (e, o))
        print("};")


if __name__ == "__main__":
    main()
