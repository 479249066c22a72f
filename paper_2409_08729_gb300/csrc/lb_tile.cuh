// lb_tile.cuh -- one tile of pairs through the whole path, in one thread block.
//
// The paper sorts all pairs by expression before launching one thread per
// pair (Sec. 4.3), so that warps do not diverge.  Here the grouping happens
// on chip, per tile of NT * LB_ITEMS pairs (NT threads per block):
//   tile_bin   loads the tile (coalesced, two pairs per load instruction),
//              handles domain edges, classifies the rest (Table "input
//              ranges") and sorts the pairs into one shared-memory list by
//              key: the region, and for mu_20 and the power series the
//              estimated term count too, so each region's pairs form one
//              contiguous range of the list, ordered by term count;
//   tile_eval  evaluates the per-thread expressions: warps take 32-pair
//              chunks of the list from shared counters, region by region,
//              so every warp runs a single expression at a time, on lanes
//              that need about the same number of terms; then stores the
//              tile's results coalesced (two per store instruction).
// The per-call kernels (logbessel.cu) and the persistent serving kernel
// (lb_serve.cu) are both built from these two steps; FP64 K pairs of the
// fallback region are left in the list for the K integral.
#pragma once

#include "lb_expr.cuh"
#include "lb_expr32.cuh"
#include "lb_kint.cuh"
#include "lb_ktrap.cuh"

// Threads per block of the serving kernel and of the K-integral and
// auxiliary kernels; the per-call tile kernel takes its own block size
// (LB_TILE_THREADS in logbessel.cu).  A tile holds LB_ITEMS pairs per thread.
#ifndef LB_THREADS
#define LB_THREADS 256
#endif
#ifndef LB_ITEMS
#define LB_ITEMS 4
#endif
#define LB_TILE (LB_THREADS * LB_ITEMS)            // tile of the serving kernel

namespace lb {

// Checked build (-DLB_CHECKS, liblogbessel_checks.so): every index into the
// tile's shared list, into the K-integral queue, and every pair offset read
// back from the queue is checked against its bound before use; a failed
// check sets a bit of lb_check_status (1 list write, 2 list read, 4 queue
// write, 8 queue count above the capacity, 16 pair offset beyond the chunk,
// 32 queue key out of range) and the access is skipped or clamped.  It
// stands in for a memory checker: the kernels record where an index left
// its buffer instead of faulting.  Release builds compile the checks out.
#ifdef LB_CHECKS
static __device__ unsigned int lb_check_status;
#define LB_CHECK(cond, bit) ((cond) || (atomicOr(&lb_check_status, (unsigned)(bit)), false))
#else
#define LB_CHECK(cond, bit) true
#endif

// List keys.  mu_20 (FP64) takes one key per term count n = 1..20 (mu_counts);
// the uniform expansions U_13 .. U_4 share one range of ten keys, by the
// pair's number of terms, largest first (in FP64 at most the region's,
// uni_terms); the power series one key per band of x, log-spaced,
// 2 log2(1 + x) (its term count grows with x: rank correlation 0.98), because
// its exact count is a loop of up to 90 steps that is cheaper once per
// 32-pair chunk than once per item round.  So each region's pairs come
// ordered by the number of terms their lanes sum.  Keys of a region are
// adjacent; regions come in the order of their list ranges.
enum TileKey {
  KEY_MU20 = 0,                  // .. KEY_MU20 + 19
  KEY_U = 20,                    // .. KEY_U + 9: 13 .. 4 terms
  KEY_FB = 30,                   // .. KEY_FB + 8: power series (I), K integral (K)
  KEY_MU3 = 39,
  NKEYS = 40
};

__host__ __device__ constexpr int region_key_first(int r) {
  return r == R_MU20 ? KEY_MU20 : r == R_FALLBACK ? KEY_FB : r == R_MU3 ? KEY_MU3 : KEY_U;
}
__host__ __device__ constexpr int region_key_end(int r) {
  return r == R_MU20 ? KEY_MU20 + 20 : r == R_FALLBACK ? KEY_FB + 9 : r == R_MU3 ? KEY_MU3 + 1 : KEY_U + 10;
}
// Terms of a uniform expansion region.
__host__ __device__ constexpr int region_terms(int r) { return r == R_U4 ? 4 : r == R_U6 ? 6 : r == R_U9 ? 9 : 13; }

// One tile of NT * IT pairs in the shared memory of a block of NT threads.
template <typename T, int NT, int IT>
struct TileShared {
  static constexpr int kTile = NT * IT;
  T sv[kTile];
  union {                                          // a pair's result replaces its argument
    T sx[kTile];
    T sres[kTile];                                 // results, stored coalesced at the end of the tile
  };
  uint16_t list[kTile];                            // tile offsets of the pairs to evaluate, sorted by key
  uint8_t nt[kTile];                               // term count (uniform expansions), class (K fallback)
  uint8_t keep[kTile];                             // 1: sres holds this pair's result
  uint16_t wcount[IT][NT / 32][NKEYS];       // pairs per (item round, warp, key), then offsets
  int kbeg[NKEYS + 1];                             // start of each key's range in list
  int next_chunk[8];                               // per region: next chunk of 32 pairs to hand out (tile_eval)
  unsigned int qbase;
  // the range of region r in list
  __device__ __forceinline__ int rbeg(int r) const { return kbeg[region_key_first(r)]; }
  __device__ __forceinline__ int rend(int r) const { return kbeg[region_key_end(r)]; }
  __device__ __forceinline__ int rcount(int r) const { return rend(r) - rbeg(r); }
};

template <int KIND, bool DX, typename T>
__device__ __forceinline__ bool tile_special(T v, T x, T* r) {
  if constexpr (sizeof(T) == 8) {
    return DX ? special_dx<KIND>(v, x, r) : special_value<KIND>(v, x, r);
  } else {
    return special_value32<KIND>(v, x, r);
  }
}

template <int KIND, bool DX, typename T>
__device__ __forceinline__ int tile_classify(T v, T x, int mode) {
  if constexpr (sizeof(T) == 8) return classify(v, x, mode, DX ? WIDE_NONE : (KIND == KIND_K ? WIDE_K : WIDE_I));
  else return classify32(v, x, mode, DX ? WIDE_NONE : (KIND == KIND_K ? WIDE_K : WIDE_I));
}

// The 16 KB table of kt_exp2_q58 in shared memory (random lookups cost a few
// bank conflicts there, up to 32 cache-line accesses in global memory).  All
// NT threads of the block call it; the caller synchronizes.  16 bytes at a
// time: both arrays are declared with that alignment.
template <int NT>
__device__ __forceinline__ void kt_load_table(unsigned long long* tab) {
  for (int i = 2 * threadIdx.x; i < 2048; i += 2 * NT)
    *reinterpret_cast<ulonglong2*>(tab + i) = *reinterpret_cast<const ulonglong2*>(lb_kt_exp2 + i);
}

// One pair per lane of region r (R_U13 stands for every U_K): n is the lane's
// term count (mu_counts, U_K's terms, series_terms).  so (FP64 values only):
// the constants of a call whose pairs all have one order, or NULL; tab: the
// table of kt_exp2_q58 (K integral).
template <int KIND, bool DX, typename T, bool SO>
__device__ __forceinline__ T tile_expr(int r, T v, T x, int n, const ScalarOrder* so,
                                       const unsigned long long* tab) {
  if constexpr (sizeof(T) == 4) {
    switch (r) {
      case R_MU20: return mu_expr32<KIND, 20>(v, x);
      case R_MU3: return mu_expr32<KIND, 3>(v, x);
      case R_FALLBACK: return (KIND == KIND_I) ? series_log_i32(v, x) : kt_log_k32(v, x);
      default:
        return n == 4 ? u_expr32<KIND, 4>(v, x) : n == 6 ? u_expr32<KIND, 6>(v, x)
             : n == 9 ? u_expr32<KIND, 9>(v, x) : u_expr32<KIND, 13>(v, x);
    }
  } else if constexpr (DX) {
    switch (r) {
      case R_MU20: return mu_dx_n<KIND>(v, x, n, 20);
      case R_MU3: return mu_dx_n<KIND>(v, x, n, 3);
      case R_FALLBACK: return (KIND == KIND_I) ? series_dx_n(v, x, n) : kt_eval<true>(v, x, n, tab);
      default: {
        const int Kmax = __reduce_max_sync(0xffffffffu, n);
        const double s = fma(v, v, x * x);
        return uni_ok(s, x) ? u_dx_fx(KIND, v, x, s, n, Kmax) : u_dx<KIND>(v, x, n);
      }
    }
  } else {
    switch (r) {
      case R_MU20:
        if constexpr (SO) return mu_expr_so<KIND>(*so, x, n);
        else return mu_expr_n<KIND>(v, x, n, 20);
      case R_MU3: return mu_expr_n<KIND>(v, x, n, 3);
      case R_FALLBACK:
        if constexpr (KIND == KIND_K) return kt_eval<false>(v, x, n, tab);
        else if constexpr (SO) return series_so(*so, x, n);
        else return series_log_i_n(v, x, n);
      default: {
        const double s = fma(v, v, x * x);
        if constexpr (SO)
          if (so->uk) return uni_ok(s, x) ? so_u(KIND, so->u, 3 * so->uk, v, x, s) : u_expr<KIND>(v, x, n);
        const int Kmax = __reduce_max_sync(0xffffffffu, n);
        return uni_ok(s, x) ? u_fx(KIND, v, x, s, n, Kmax) : u_expr<KIND>(v, x, n);
      }
    }
  }
}

// List key of a classified pair, and in *n the term count of a uniform
// expansion or the class of a K fallback pair (0 otherwise).
// KIN: FP64 K fallback pairs are evaluated in the tile, by class (kt_class,
// costliest first).
template <int KIND, bool DX, typename T, bool KIN>
__device__ __forceinline__ int tile_key(int r, T v, T x, int* n) {
  *n = 0;
  if (r == R_MU20) {
    if constexpr (sizeof(T) == 8) return KEY_MU20 + (mu_counts(f32_cut(v), f32_cut(x)) & 255) - 1;
    return KEY_MU20;
  }
  if (r == R_MU3) return KEY_MU3;
  if (r == R_FALLBACK) {
    if (KIND == KIND_I) return KEY_FB + min(8, (int)(2.0f * __log2f(1.0f + (sizeof(T) == 8 ? f32_cut((double)x) : (float)x))));
    if constexpr (KIN) {
      *n = kt_class(v, x, DX);
      return KEY_FB + *n;
    }
    return KEY_FB;
  }
  int K = region_terms(r);
  if constexpr (sizeof(T) == 8) {
    const float vf = f32_cut(v), xf = f32_cut(x), s = fmaf(vf, vf, xf * xf);
    K = DX ? uni_terms_dx(s, K) : uni_terms(s, K);
  }
  *n = K;
  return KEY_U + 13 - K;
}

// Tile offset of item round `it` of thread `tid`: each thread handles two
// adjacent pairs per pair of rounds, so it loads and stores them with one
// 16-byte (FP64) or 8-byte (FP32) instruction.
// IT = 1: one pair per thread.
template <int NT, int IT>
__device__ __forceinline__ int tile_offset(int it, int tid) {
  return IT == 1 ? tid : (it >> 1) * (2 * NT) + 2 * tid + (it & 1);
}

template <typename T>
struct Vec2;
template <>
struct Vec2<double> { typedef double2 type; };
template <>
struct Vec2<float> { typedef float2 type; };

// Load, edge-handle, classify and sort pairs [t0, min(t0 + NT * IT, n)).
// All threads of the block call it; it ends with a barrier.  The list is
// ordered by (key, item round, warp, lane), from one warp match per item
// and a per-key prefix over (item round, warp): the order, and so the warp
// mates of every pair, do not depend on scheduling.
// v0: the order of every pair when v_stride is 0 (v is not read then).
template <int KIND, bool DX, typename T, bool KIN, int NT, int IT>
__device__ __forceinline__ void tile_bin(TileShared<T, NT, IT>& S, const T* __restrict__ v, int64_t v_stride, T v0,
                                         const T* __restrict__ x, int64_t t0, int64_t n, int mode,
                                         int forced_region) {
  typedef typename Vec2<T>::type T2;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const unsigned int lt = (1u << lane) - 1u;
  // the pair offsets t0 are multiples of the tile size, so aligned bases keep every pair of loads aligned
  const bool vec = ((reinterpret_cast<uintptr_t>(x) | (v_stride ? reinterpret_cast<uintptr_t>(v) : 0)) &
                    (2 * sizeof(T) - 1)) == 0;
  T vv[IT], xx[IT];
  if constexpr (IT == 1) {
    const int64_t i = t0 + tid;
    xx[0] = i < n ? x[i] : T(1);
    vv[0] = i < n ? (v_stride ? v[i] : v0) : T(0);
  } else {
#pragma unroll
    for (int h = 0; h < IT / 2; ++h) {
      const int li = tile_offset<NT, IT>(2 * h, tid);
      const int64_t i = t0 + li;
      if (vec && i + 1 < n) {
        const T2 xv = *reinterpret_cast<const T2*>(x + i);
        xx[2 * h] = xv.x;
        xx[2 * h + 1] = xv.y;
        if (v_stride) {
          const T2 vw = *reinterpret_cast<const T2*>(v + i);
          vv[2 * h] = vw.x;
          vv[2 * h + 1] = vw.y;
        } else {
          vv[2 * h] = vv[2 * h + 1] = v0;
        }
      } else {
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          xx[2 * h + e] = (i + e < n) ? x[i + e] : T(1);
          vv[2 * h + e] = (i + e < n) ? (v_stride ? v[i + e] : v0) : T(0);
        }
      }
    }
  }
  int key[IT], rank[IT];
#pragma unroll
  for (int it = 0; it < IT; ++it) {
    const int li = tile_offset<NT, IT>(it, tid);
    const int64_t i = t0 + li;
    int k = NKEYS;                                 // NKEYS: no list entry
    uint8_t keep = 0;
    if (i < n) {
      T vi = vv[it];
      const T xi = xx[it];
      if constexpr (KIND == KIND_K) {
        if constexpr (sizeof(T) == 8) vi = __longlong_as_double(__double_as_longlong(vi) & 0x7fffffffffffffffLL);
        else vi = fabsf(vi);
      }
      T sp;
      if (tile_special<KIND, DX, T>(vi, xi, &sp)) {
        S.sres[li] = sp;
        keep = 1;
      } else {
        S.sv[li] = vi;
        S.sx[li] = xi;
        const int r = forced_region >= 0 ? forced_region : tile_classify<KIND, DX, T>(vi, xi, mode);
        int nterm;
        k = tile_key<KIND, DX, T, KIN>(r, vi, xi, &nterm);
        S.nt[li] = (uint8_t)nterm;
        keep = (KIND == KIND_K && sizeof(T) == 8 && !KIN && r == R_FALLBACK) ? 0 : 1;   // queued pairs are stored later
      }
    }
    S.keep[li] = keep;
    // pairs of the same key in this warp: count and rank by lane
    for (int kk = lane; kk < NKEYS; kk += 32) S.wcount[it][warp][kk] = 0;
    __syncwarp();
    const unsigned int m = __match_any_sync(0xffffffffu, k);
    rank[it] = __popc(m & lt);
    if (k < NKEYS && rank[it] == 0) S.wcount[it][warp][k] = (uint16_t)__popc(m);
    key[it] = k;
  }
  __syncthreads();
  // exclusive prefix per key over (item round, warp); the key's total to kbeg
  if (tid < NKEYS) {
    int acc = 0;
    for (int it = 0; it < IT; ++it)
      for (int w = 0; w < NT / 32; ++w) {
        const int c = S.wcount[it][w][tid];
        S.wcount[it][w][tid] = (uint16_t)acc;
        acc += c;
      }
    S.kbeg[tid + 1] = acc;
  }
  __syncthreads();
  // exclusive scan of the key totals (one warp)
  if (warp == 0) {
    int a = S.kbeg[lane + 1], b = lane + 33 <= NKEYS ? S.kbeg[lane + 33] : 0;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int ua = __shfl_up_sync(0xffffffffu, a, o), ub = __shfl_up_sync(0xffffffffu, b, o);
      if (lane >= o) { a += ua; b += ub; }
    }
    const int tot_a = __shfl_sync(0xffffffffu, a, 31);
    __syncwarp();
    S.kbeg[lane + 1] = a;
    if (lane + 33 <= NKEYS) S.kbeg[lane + 33] = b + tot_a;
    if (lane == 0) S.kbeg[0] = 0;
  }
  if (tid < 8) S.next_chunk[tid] = 0;
  __syncthreads();
#pragma unroll
  for (int it = 0; it < IT; ++it)
    if (key[it] < NKEYS) {
      const int pos = S.kbeg[key[it]] + S.wcount[it][warp][key[it]] + rank[it];
      if (LB_CHECK(pos >= 0 && pos < (NT * IT), 1u)) S.list[pos] = (uint16_t)tile_offset<NT, IT>(it, tid);
    }
  __syncthreads();
}

// von Mises-Fisher log-normaliser (paper Sec. 6.3):
//   log C_d(k) = (d/2 - 1) log k - (d/2) log(2 pi) - log I_{d/2-1}(k),
// from f = log I_{d/2-1}(k) (or, for DX, f = d/dk log I_{d/2-1}, giving
// d/dk log C_d = (d/2-1)/k - I'/I).
// At k = 0: log C_d(0) = lgamma(d/2) - log 2 - (d/2) log pi, the limit of
// I_nu(k) ~ (k/2)^nu / Gamma(nu + 1).
template <bool DX>
__device__ __forceinline__ double vmf_form(double d, double k, double f) {
  const double nu = 0.5 * d - 1.0;
  if (DX) return (k == 0.0) ? 0.0 : (k < 1e300 ? kt_div(nu, k) : nu / k) - f;
  if (k == 0.0) return lgamma(0.5 * d) - 0.6931471805599453 - 0.5 * d * 1.1447298858494002;
  return fma(nu, ix_log_call(k), -0.5 * d * 1.8378770664093453) - f;
}

// The chunks (32 pairs, one warp each) of region R's range of the list,
// handed out from a shared counter: a warp that runs out moves on to the
// next region while the others finish this one.  Lanes past the end of the
// range recompute the chunk's first entry and do not keep it.  `so` (FP64
// values only) holds the constants of a call whose pairs all have one
// order, or is NULL.
template <int KIND, bool DX, typename T, bool SO, int R, int NT, int IT>
__device__ __forceinline__ void tile_eval_region(TileShared<T, NT, IT>& S, int lane, const ScalarOrder* so) {
  const int b0 = S.rbeg(R), c = S.rend(R) - b0;
  const int nch = (c + 31) >> 5;
  for (;;) {
    int id = 0;
    if (lane == 0) id = atomicAdd(&S.next_chunk[R], 1);
    id = __shfl_sync(0xffffffffu, id, 0);
    if (id >= nch) break;
    const int j0 = id << 5, j = j0 + lane;
    bool ok = j < c;
    int jl = b0 + (ok ? j : j0);
    if (!LB_CHECK(jl >= 0 && jl < (NT * IT), 2u)) {
      jl = 0;                                      // clamped: the warp still runs the expression together
      ok = false;
    }
    const int li = S.list[jl];
    const T v = SO ? (T)so->v : S.sv[li], x = S.sx[li];
    int n = S.nt[li];
    if constexpr (sizeof(T) == 8 && (R == R_MU20 || R == R_MU3)) n = mu_counts(f32_cut(v), f32_cut(x));
    if constexpr (sizeof(T) == 8 && KIND == KIND_I && R == R_FALLBACK) n = series_terms(f32_cut(v), f32_cut(x));
    const T val = tile_expr<KIND, DX, T, SO>(R, v, x, n, so, nullptr);
    __syncwarp();                                  // every lane has read its arguments (sres is sx)
    if (ok) S.sres[li] = val;
  }
}

// The K fallback pairs of a tile, in chunks of 32 pairs of one class: with
// few pairs per tile the chunks are not full, but run side by side on the
// block's warps instead of one class after another in one warp.
template <bool DX, int NT, int IT>
__device__ __forceinline__ void tile_eval_kint(TileShared<double, NT, IT>& S, int lane, const unsigned long long* tab) {
  for (;;) {
    int id = 0;
    if (lane == 0) id = atomicAdd(&S.next_chunk[R_FALLBACK], 1);
    id = __shfl_sync(0xffffffffu, id, 0);
    int c = 0, b = 0, e = 0;
#pragma unroll 1
    for (; c < 6; ++c) {
      b = S.kbeg[KEY_FB + c];
      e = S.kbeg[KEY_FB + c + 1];
      const int nch = (e - b + 31) >> 5;
      if (id < nch) break;
      id -= nch;
    }
    if (c == 6) break;
    const int j = b + (id << 5) + lane;
    if (j < e) {
      const int li = S.list[j];
      S.sres[li] = kt_eval<DX>(S.sv[li], S.sx[li], c, tab);   // sres is sx: read before written, by this lane alone
    }
    __syncwarp();
  }
}

// Per-thread expressions, region by region, costliest first (so that the
// last chunks of a tile are cheap and the warps reach the closing barrier
// close together); every warp runs a single expression at a time, and the
// result of a pair does not depend on which warp takes its chunk.  Then the
// tile's results (domain edges included) are stored, two pairs per
// instruction where both are kept and the buffer is aligned.  The FP64 K fallback
// pairs are left to the K integral: neither evaluated nor stored (so out may
// equal x: their arguments stay in place for it).  Ends with a barrier.
// vmf_d >= 0 (FP64 log I and its derivative only): the von Mises-Fisher form
// of the result in dimension vmf_d (vmf_form) is stored instead.
template <int KIND, bool DX, typename T, bool SO, bool KIN, int NT, int IT>
__device__ __forceinline__ void tile_eval(TileShared<T, NT, IT>& S, T* __restrict__ out, int64_t t0, int64_t n,
                                          const ScalarOrder* so = nullptr, const T* __restrict__ x = nullptr,
                                          double vmf_d = -1.0, const unsigned long long* tab = nullptr) {
  typedef typename Vec2<T>::type T2;
  const int tid = threadIdx.x, lane = tid & 31;
  if constexpr (KIN) tile_eval_kint<DX>(S, lane, tab);
  else if (KIND == KIND_I || sizeof(T) == 4) tile_eval_region<KIND, DX, T, SO, R_FALLBACK>(S, lane, so);
  tile_eval_region<KIND, DX, T, SO, R_U13>(S, lane, so);
  tile_eval_region<KIND, DX, T, SO, R_MU20>(S, lane, so);
  tile_eval_region<KIND, DX, T, SO, R_MU3>(S, lane, so);
  __syncthreads();
  const bool vec = (reinterpret_cast<uintptr_t>(out) & (2 * sizeof(T) - 1)) == 0;
#pragma unroll
  for (int h = 0; h < (IT + 1) / 2; ++h) {
    const int li = tile_offset<NT, IT>(2 * h, tid);
    const int64_t i = t0 + li;
    const bool k0 = i < n && S.keep[li], k1 = IT > 1 && i + 1 < n && S.keep[li + (IT > 1)];
    if constexpr (sizeof(T) == 8 && KIND == KIND_I) {
      if (vmf_d >= 0.0) {
        if (k0) S.sres[li] = vmf_form<DX>(vmf_d, x[i], S.sres[li]);
        if (k1) S.sres[li + 1] = vmf_form<DX>(vmf_d, x[i + 1], S.sres[li + 1]);
      }
    }
    if (vec && k0 && k1) {
      T2 r;
      r.x = S.sres[li];
      r.y = S.sres[li + 1];
      *reinterpret_cast<T2*>(out + i) = r;
    } else {
      if (k0) out[i] = S.sres[li];
      if (k1) out[i + 1] = S.sres[li + 1];
    }
  }
  __syncthreads();
}

// K integral of a batch of up to 32 pairs by one warp (the paper's Simpson
// rule): lane e holds pair e; each lane computes its pair's prefactor, then
// the warp evaluates the integrals one pair at a time with the nodes spread
// over the lanes.
__device__ __forceinline__ double kint_warp_batch(double vi, double xi, int m, int lane) {
  const double pre = kint_prefactor(vi, xi);
  double mine = 0;
  for (int e = 0; e < m; ++e) {
    const double ve = __shfl_sync(0xffffffffu, vi, e);
    const double xe = __shfl_sync(0xffffffffu, xi, e);
    const double li = kint_log_simpson(ve, xe, lane);
    if (lane == e) mine = li;
  }
  return pre + mine;
}

// One pair per warp, tight mode (FP64): for calls with too few pairs for the
// tiles to fill the GPU.  Every lane holds the pair (i, the same for the warp)
// and computes the same.  One kernel and no queue; tab: 16 KB of shared memory
// for the K integral's table (filled if a pair of the block needs it).
template <int KIND, bool DX, int NT>
__device__ __forceinline__ void warp_pair64(const double* __restrict__ v, int64_t v_stride, double v0,
                                            const double* __restrict__ x, double* __restrict__ out, int64_t i,
                                            bool valid, double vmf_d, unsigned long long* tab) {
  double vi = valid ? (v_stride ? v[i] : v0) : 1.0;
  const double xi = valid ? x[i] : 1.0;
  if constexpr (KIND == KIND_K) vi = fabs(vi);
  double val = 0.0;
  int r = R_SPECIAL, n = 0;
  if (valid && !tile_special<KIND, DX, double>(vi, xi, &val)) {
    r = tile_classify<KIND, DX, double>(vi, xi, MODE_TIGHT);
    tile_key<KIND, DX, double, true>(r, vi, xi, &n);
    if (r == R_MU20) n = mu_counts(f32_cut(vi), f32_cut(xi));
    if (KIND == KIND_I && r == R_FALLBACK) n = series_terms(f32_cut(vi), f32_cut(xi));
    if (r != R_MU20 && r != R_FALLBACK) r = R_U13;         // every uniform expansion
  }
  if constexpr (KIND == KIND_K) {
    if (__syncthreads_or(r == R_FALLBACK)) {
      kt_load_table<NT>(tab);
      __syncthreads();
    }
  }
  if (r != R_SPECIAL) val = tile_expr<KIND, DX, double, false>(r, vi, xi, n, nullptr, tab);
  if constexpr (KIND == KIND_I) {
    if (valid && vmf_d >= 0.0) val = vmf_form<DX>(vmf_d, xi, val);
  }
  if (valid && (threadIdx.x & 31) == 0) out[i] = val;
}

// FP32 pairs in tight mode (log I or log K).  Each warp works by itself, with
// no block barrier: it takes slices of 32 VEC adjacent pairs (VEC = 4: one
// 16-byte load of v and x per lane), evaluates u_all32 where
// r^2 = v^2 + x^2 >= 14^2, and stores; the other pairs (series or K integral)
// go to a list of the warp in shared memory, and whenever it holds 256 it is
// sorted by an estimate of their loops' length (16 keys) and evaluated, 32
// at a time.  Nothing else is binned: binning every pair by region, as the
// FP64 tiles do, costs more instructions than the one merged expansion.  A
// pair's result depends on the pair alone.  The listed pairs' arguments are
// read again from global memory; their outputs are not written before where out
// is x or v.
constexpr int kList32 = 256 + 128;                         // entries before a flush, and one slice's
struct Warp32 {
  uint32_t raw[kList32], list[kList32];                    // offsets from the base of v, x and out
  uint8_t rkey[kList32];
  int count[16];
};

// The pairs that warp_pairs32 does not list or evaluate in line: domain edges,
// v or x above 1e18, x below kTinyX32.  Called, so that the loop's code stays
// small.
template <int KIND>
static __device__ __noinline__ float edge32(float v, float x) {
  float r;
  if (special_value32<KIND>(v, x, &r)) return r;
  if (v <= 1e18f && x < 1.0f) {
    if (v * v >= kAllR2) return u_all32<true>(KIND, v, x, v * v);
    return KIND == KIND_I ? series_all32(v, x) : kt_small32(v, x);
  }
  const int g = classify32(v, x, MODE_TIGHT, KIND == KIND_K ? WIDE_K : WIDE_I);
  return g == R_MU20 ? mu_expr32<KIND, 20>(v, x) : u_expr32<KIND, 4>(v, x);
}

// Sort key of a listed pair, 0 .. 15, in order of decreasing work.
template <int KIND>
__device__ __forceinline__ int key32(float v, float x) {
  if (KIND == KIND_I) return 15 - min(15, (int)(3.8f * __log2f(1.0f + x)));   // term count grows with x
  if (x < 0x1p-9f) return 15 - min(3, (int)(0.25f * v));
  const float a2 = v + sqrtf(fmaf(v, v, x * x));
  const float left = fminf(__log2f(2.0f + __fdividef(36.0f * a2, x * x)), __fdividef(18.0f + 0.5f * a2, 0.7f * v));
  const int m = kt_step32(v, x);                           // left (2 + m) nodes a side
  return 4 * m + 3 - max(0, min(3, (int)((left - 3.0f) * 0.25f)));
}

// Sort the warp's list (cnt entries) and evaluate it; all of it, or (last =
// false) whole chunks of 32 only.  Returns the entries left in the list.
template <int KIND>
__device__ __forceinline__ int flush32(Warp32& W, int cnt, bool last, const float* __restrict__ v, int64_t v_stride,
                                       const float* __restrict__ x, float* __restrict__ out) {
  const int lane = threadIdx.x & 31;
  if (lane < 16) W.count[lane] = 0;
  __syncwarp();
  for (int j = lane; j < cnt; j += 32) {
    const int64_t i = W.raw[j];
    const float vi = v[i * v_stride];
    const int k = key32<KIND>(KIND == KIND_K ? fabsf(vi) : vi, x[i]);
    W.rkey[j] = (uint8_t)k;
    atomicAdd(&W.count[k], 1);
  }
  __syncwarp();
  const int c = lane < 16 ? W.count[lane] : 0;
  int p = c;
#pragma unroll
  for (int o = 1; o < 16; o <<= 1) {
    const int u = __shfl_up_sync(0xffffffffu, p, o);
    if (lane >= o) p += u;
  }
  if (lane < 16) W.count[lane] = p - c;                    // where each key's entries begin
  __syncwarp();
  for (int j = lane; j < cnt; j += 32) {
    const int k = W.rkey[j], pos = atomicAdd(&W.count[k], 1);
    if (LB_CHECK(pos < kList32, 1u)) W.list[pos] = W.raw[j];
  }
  __syncwarp();
  const int m = last ? cnt : cnt & ~31;
  for (int j = lane; j < m; j += 32) {
    const int64_t i = W.list[j];
    const float vi = v[i * v_stride], xi = x[i];
    out[i] = KIND == KIND_I ? series_all32(vi, xi) : kt_log_k32(fabsf(vi), xi);
  }
  __syncwarp();
  if (lane < cnt - m) W.raw[lane] = W.list[m + lane];
  __syncwarp();
  return cnt - m;
}

// This warp's share of the pairs [begin, end): slices warp, warp + nwarps, ...
// Offsets fit 32 bits (the caller's pointers are based accordingly).
template <int KIND, int VEC>
__device__ __forceinline__ void warp_pairs32(Warp32& W, const float* __restrict__ v, int64_t v_stride,
                                             const float* __restrict__ x, float* __restrict__ out, int64_t begin,
                                             int64_t end, int64_t warp, int64_t nwarps) {
  const int lane = threadIdx.x & 31;
  const unsigned lt = (1u << lane) - 1u;
  const float v0 = v_stride ? 0.0f : v[0];
  const bool in_place = out == x || out == v;
  int cnt = 0;                                             // entries in the list (warp-uniform)
  for (int64_t s = begin + warp * (32 * VEC); s < end; s += nwarps * (32 * VEC)) {
    const int64_t i = s + lane * VEC;
    float vv[VEC], xx[VEC], rr[VEC];
    const bool whole = VEC == 4 && i + 3 < end;
    if (whole) {
      const float4 a = *reinterpret_cast<const float4*>(x + i);
      xx[0] = a.x;
      if (VEC == 4) { xx[1 % VEC] = a.y; xx[2 % VEC] = a.z; xx[3 % VEC] = a.w; }
      if (v_stride) {
        const float4 b = *reinterpret_cast<const float4*>(v + i);
        vv[0] = b.x;
        if (VEC == 4) { vv[1 % VEC] = b.y; vv[2 % VEC] = b.z; vv[3 % VEC] = b.w; }
      } else {
#pragma unroll
        for (int e = 0; e < VEC; ++e) vv[e] = v0;
      }
    } else {
#pragma unroll
      for (int e = 0; e < VEC; ++e) {
        xx[e] = i + e < end ? x[i + e] : 50.0f;
        vv[e] = i + e < end ? (v_stride ? v[i + e] : v0) : 1.0f;
      }
    }
    unsigned fb = 0;                                       // bit e: pair e goes to the list
#pragma unroll
    for (int e = 0; e < VEC; ++e) {
      const float xi = xx[e], vi = KIND == KIND_K ? fabsf(vv[e]) : vv[e];
      // one test for the domain edges, squares out of range and quotients that underflow
      if (!(xi >= kTinyX32 && xi <= 1e18f && vi >= 0.0f && vi <= 1e18f)) {
        rr[e] = edge32<KIND>(vi, xi);
      } else {
        const float s2 = fmaf(vi, vi, xi * xi);
        if (s2 < kAllR2) fb |= 1u << e;
        rr[e] = u_all32<false>(KIND, vi, xi, s2);
      }
    }
    // a listed pair's result is written after this by the same warp; its slot
    // may hold anything until then, except its argument or its order when out is x or v
    if (whole && (fb == 0 || !in_place)) {
      if (VEC == 4) *reinterpret_cast<float4*>(out + i) = make_float4(rr[0], rr[1 % VEC], rr[2 % VEC], rr[3 % VEC]);
    } else {
#pragma unroll
      for (int e = 0; e < VEC; ++e)
        if (i + e < end && !((fb >> e) & 1u)) out[i + e] = rr[e];
    }
#pragma unroll
    for (int e = 0; e < VEC; ++e) {
      const bool f = ((fb >> e) & 1u) && i + e < end;
      const unsigned m = __ballot_sync(0xffffffffu, f);
      const int b = cnt + __popc(m & lt);
      if (f && LB_CHECK(b < kList32, 1u)) W.raw[b] = (uint32_t)(i + e);
      cnt += __popc(m);
    }
    if (cnt >= 256) cnt = flush32<KIND>(W, cnt, false, v, v_stride, x, out);
  }
  if (cnt > 0) flush32<KIND>(W, cnt, true, v, v_stride, x, out);
}

}  // namespace lb
