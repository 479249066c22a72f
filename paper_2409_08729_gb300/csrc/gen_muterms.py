"""Generates muterms_table.h: term counts of the large-argument expansion.

    python3 gen_muterms.py > muterms_table.h

S = 1 + sum_k +-t_k, t_k = prod_{j<=k} |A - (2j-1)^2 w| / j with
A = v^2/(2x) and w = 1/(8x).  Per cell of (A, w), n: the smallest count <= 20
after which the terms stay below 2^-56, and h: the smallest k from which they
stay below 1e-3 (20 where there is none), each the largest over a grid of
points of the cell.  Cells are half octaves, [2^e, 1.5 2^e) and
[1.5 2^e, 2^(e+1)); the first row and column stand for everything below, the
last for everything above, with both counts 20.
"""
import numpy as np

A_LO, A_CELLS = -24, 54      # A from 2^-24 to 2^3
W_LO, W_CELLS = -27, 40      # w from 2^-27 to 2^-7
K = 20


def counts(A, w):
    t = np.ones_like(A)
    n = np.full(A.shape, 1)
    h = np.full(A.shape, 1)
    for k in range(1, K + 1):
        t = t * np.abs(A - (2 * k - 1) ** 2 * w) / k
        # the terms up to k: counts are one past the last term above the bound
        n = np.where(t >= 1.4e-17, k + 1, n)
        h = np.where(t >= 1e-3, k + 1, h)
    return np.minimum(n, K), np.minimum(h, K)


def cell(i, lo):
    e, half = divmod(i, 2)
    a = 2.0 ** (lo + e) * (1.5 if half else 1.0)
    b = 2.0 ** (lo + e) * (2.0 if half else 1.5)
    return a, b


def main():
    print("// Generated by gen_muterms.py: do not edit.")
    print("#pragma once")
    print("#define LB_MUT_A_CELLS %d   // + 1 column for A above" % A_CELLS)
    print("#define LB_MUT_W_CELLS %d   // + 1 row for w above" % W_CELLS)
    print("#define LB_MUT_A_BASE %d   // float bits >> 22 of the first cell" % ((127 + A_LO) * 2))
    print("#define LB_MUT_W_BASE %d" % ((127 + W_LO) * 2))
    print("// n | h << 8; [row of w][column of A]")
    print("LB_MUT_TABLE unsigned short lb_mut[%d] = {" % ((W_CELLS + 1) * (A_CELLS + 1)))
    for iw in range(W_CELLS + 1):
        row = []
        for ia in range(A_CELLS + 1):
            if iw == W_CELLS or ia == A_CELLS:
                n, h = K, K
            else:
                wa, wb = cell(iw, W_LO)
                aa, ab = cell(ia, A_LO)
                w = np.concatenate([[0.0] if iw == 0 else [], np.linspace(wa, wb, 33)])
                A = np.concatenate([[0.0] if ia == 0 else [], np.linspace(aa, ab, 65)])
                AA, WW = np.meshgrid(A, w)
                n, h = counts(AA, WW)
                n, h = int(n.max()), int(h.max())
            row.append("0x%04x" % (n | h << 8))
        print("    " + ", ".join(row) + ",")
    print("};")


if __name__ == "__main__":
    main()
