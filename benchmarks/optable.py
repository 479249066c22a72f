"""Algorithmic work of the evaluation kernels, for the roofline: a fixed table.

Work is the number of FP64 arithmetic operations the method performs, one
per add, subtract, multiply, fused multiply-add or compare: each is one
issue of the FP64 pipe, whose peak is 2 operations per SM per clock
(152 SMs x 2 x 2.07 GHz = 629.3 G op/s on GB300).  Calls to transcendental
and other library functions (log, exp, reciprocal, 1/sqrt, lgamma) are
counted by name and NOT priced: how a call is evaluated (here mostly on the
integer pipes) is the implementation's business, so the FP64 operations of
the method are a lower bound on the FP64-pipe work of any implementation,
and frac = (table operations) / (time x peak) is the share of the FP64
pipe's capacity that did the method's own arithmetic.

Per pair, in tight mode, with n the pair's own term count (not the warp's):

  region          general pair                  one order for the whole call
  mu_K (n terms)  2n + 8     rcp, log           n + 6     rcp, log
  U_K             K(K+1)/2 + K + 14             3K + 13 (orders above 10)
                  rsqrt, 3 log                  rsqrt, 3 log
  series (n)      4n + 7     rcp, 2 log, lgamma 2n + 5    2 log
  K integral      7 per node, 14 per pair       the same
                  exp: 1 per node, rsqrt, 2 rcp, 2 log per pair
  (x < 2^-9)      64 per pair + 2 per step of the recurrence
                  log, exp, 6 rcp, log

mu_K: per term D_k = mu w - (2k-1)^2 w (fma) and Q <- D_k Q + const (fma);
per pair mu w (3), 8x, S^2 w (2), scaling, the final fma.  With one order the
sum is a polynomial in w: one fma per term.
U_K: v^2 + x^2, r = (v^2 + x^2) / sqrt, v/r, its square, v + r, the Debye
polynomial P_k of degree k by Horner (k fmas, k = 1..K), Horner over k in 1/r
(K fmas), S^2/r (2), the difference of the logarithms, final fmas.  K is the
pair's own: its region's, or less at large r.  With one order above 10 the sum
is one polynomial in v/r of degree 3K, K the order's (3K fmas).
Series (the linear fraction of the reading of Eq. "log Iv" with a_0 as
shift): per term d_k = k(k+v) (fma), A <- d B + y A (mul, fma), B <- d B;
per pair y = x^2/4, A/B, v+1, x/2, two combining operations.  With one
order the ratios 1/(k(k+v)) are the call's: per term y r_k and one fma.
K integral (trapezoid rule about the maximum): a node forms a e^(kh) and
b e^(-kh) (two multiplications by constants), their sum, the linear term,
their difference from the maximum, the exponential, and its addition to the
sum; per pair v^2 + x^2 (2), r, r + v, x^2/(r + v) (2), v h, x^2, (r + v)/x,
the two logarithms' combination (5).  Below x = 2^-9 Temme's series: 64
operations and two per step from order mu to v.
FP32-mixed form (FP32 operations): one expansion of five terms for
r >= 14 (45), the series 5n + 30, the integral 5 per node + 14.
"""
import numpy as np

PEAK_FP64_OPS = 152 * 2 * 2.07e9       # FP64-pipe operations per second: SMs x DFMA/clk x max clock
PEAK_FP32_OPS = 152 * 128 * 2.07e9     # FP32-pipe operations per second: SMs x FP32 lanes x max clock

REGION_NAMES = {0: "mu20", 1: "u13", 2: "fallback", 4: "mu3", 5: "u4", 6: "u6", 7: "u9"}
REGION_K = {0: 20, 1: 13, 4: 3, 5: 4, 6: 6, 7: 9}      # expansion terms of each region


def mu_terms(v, x, K=20, eps=1.4e-17):
    """Terms the mu_K expression needs for each pair: the first k after which
    a term falls below eps (2^-56: the FP64 kernels' single-precision
    estimate; the FP32 form counts to 2^-24)."""
    v = np.asarray(v, dtype=np.float32)
    x = np.asarray(x, dtype=np.float32)
    mu = np.float32(4.0) * v * v
    inv8x = np.float32(1.0) / (np.float32(8.0) * x)
    t = np.ones_like(x)
    n = np.full(x.shape, K, dtype=np.int64)
    done = np.zeros(x.shape, dtype=bool)
    for k in range(1, K + 1):
        t = np.where(done, t, t * (mu - np.float32((2 * k - 1) ** 2)) * inv8x / np.float32(k))
        hit = ~done & (np.abs(t) < eps)
        n = np.where(hit, k, n)
        done |= hit
    return n


def series_terms(v, x, eps=1.4e-17):
    """Terms the power series sums for each pair (the kernels' single-precision
    estimate: past the peak index, until a term is below eps of the sum;
    2^-56 in FP64, 1.5e-8 in the FP32 form)."""
    v = np.asarray(v, dtype=np.float32)
    x = np.asarray(x, dtype=np.float32)
    y = np.float32(0.25) * x * x
    kpk = np.float32(0.5) * (np.sqrt(x * x + v * v) - v)
    term = np.ones_like(x)
    T = np.zeros_like(x)
    n = np.ones(x.shape, dtype=np.int64)
    done = np.zeros(x.shape, dtype=bool)
    for k in range(1, 91):
        active = ~done
        if not active.any():
            break
        term = np.where(active, term * y / (np.float32(k) * (np.float32(k) + v)), term)
        T = np.where(active, T + term, T)
        n = np.where(active, k, n)
        done |= active & (np.float32(k) > kpk) & (term <= np.float32(eps) * (1 + T))
    return n


def uni_terms(v, x, cap):
    """Terms of the uniform expansion (FP64 values): the region's cap, or the
    smallest K with max|P_(K+1)| / r^(K+1) <= 3e-17 r, by half octaves."""
    s = (np.asarray(v, dtype=np.float32) ** 2 + np.asarray(x, dtype=np.float32) ** 2).astype(np.float32)
    i = (s.view(np.uint32) >> 22).astype(np.int64) - (2 * (127 + 9) + 1)
    tab = np.array([13, 12, 11, 10, 9, 8, 8, 7, 7, 6, 6, 6, 5, 5, 5, 5, 4])
    return np.minimum(np.where(i < 0, 13, tab[np.clip(i, 0, 16)]), cap)


def kint_nodes(v, x, fp32=False):
    """Nodes of the tight K-integral rule of each pair (|v| given): both sides
    of the maximum in groups of m (h = ln2/m) to the first group whose last
    term is below 2^-54 (FP32: node by node to 2^-26), and the maximum; 0 for
    x < 2^-9 (Temme's series)."""
    v = np.asarray(v, dtype=np.float64)
    x = np.asarray(x, dtype=np.float64)
    if fp32:
        m = np.where(x <= 6.8 - 1.8 * v, 2, np.where(x <= 19.5 - 0.115 * v * v, 3, 4))
    else:
        m = np.where(x <= 4.5 - 1.5 * v * v, 3, np.where(x <= 17.8 - 0.28 * v * v, 4,
                                                        np.where(x <= 31 - 0.09 * v * v, 5, 6)))
    r = np.hypot(v, x)
    a = (r + v) / 2 / np.log(2)
    b = x * x / (2 * (r + v)) / np.log(2)
    cut, step = (26, 1.0 / m) if fp32 else (54, 1.0)
    total = np.ones(v.shape, dtype=np.int64)
    for p, q, sgn in ((a, b, 1.0), (b, a, -1.0)):
        live = x >= 2.0 ** -9
        for k in range(1, 400):
            if not live.any():
                break
            total += np.where(live, 1 if fp32 else m, 0)
            d = np.minimum(k * step, 500.0)
            live = live & (p * 2.0 ** d + q * 2.0 ** -d - (a + b) - sgn * v * d <= cut)
    return np.where(x >= 2.0 ** -9, total, 0)


def region_ops(region, v, x, shared=False, fp32=False):
    """Operations per pair of the per-thread expressions (tile kernel): FP64,
    or FP32 for the FP32-mixed form (term counts to single precision; its
    calls pass no order constants, so shared does not apply)."""
    shape = np.shape(x)
    shared = shared and not fp32
    if fp32:
        return 5 * series_terms(v, x, eps=1.5e-8) + 30 if region == 2 else np.full(shape, 45, dtype=np.int64)
    if region in (0, 4):
        n = mu_terms(v, x, REGION_K[region])
        return (n + 6) if (shared and region == 0) else (2 * n + 8)
    if region in REGION_K:
        K = uni_terms(v, x, REGION_K[region])
        ops = K * (K + 1) // 2 + K + 14
        return np.where(np.abs(v) > 10.0, 3 * REGION_K[region] + 13, ops) if shared else ops
    n = series_terms(v, x)
    return (2 * n + 5) if shared else (4 * n + 7)


def kint_ops(v, x, shared=False, fp32=False):
    """Operations per pair of the K integral."""
    n = kint_nodes(v, x, fp32)
    return np.where(n > 0, (5 if fp32 else 7) * n + 14, 64 + 2 * np.floor(np.asarray(v) + 0.5).astype(np.int64))


def region_calls(region, shared=False):
    """Library calls per pair (named, not priced) of each expression."""
    if region in (0, 4):
        return {"rcp": 1, "log": 1}
    if region in REGION_K:
        return {"rsqrt": 1, "log": 3}
    return {"log": 2} if shared else {"rcp": 1, "log": 2, "lgamma": 1}
