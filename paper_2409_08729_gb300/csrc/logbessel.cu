// logbessel.cu -- kernels and C ABI of the GB300 log-Bessel library.
//
// Pipeline for one call (paper Sec. 4.3 sorts the pairs by expression before
// launch so that warps do not diverge; here the grouping is done on chip):
//
//   1. lb_tiles_kernel: persistent CTAs walk tiles of 256 to 2048 pairs (by
//      the size of the call).  Each thread loads its pairs (coalesced),
//      handles domain edges, and classifies the rest (Table "input ranges").
//      The tile's pairs are binned per region into shared-memory index lists;
//      the warps take 32-pair chunks of the lists from shared counters, so
//      every warp runs one expression (mu_20, U_K, power series) at a time.
//      K pairs of the fallback region are evaluated in the tile (calls below
//      2^17 pairs) or appended to a global queue.
//   2. lb_ktrap_kernel (tight FP64): one thread per queued K pair evaluates the
//      integral by the trapezoid rule (lb_ktrap.cuh); lb_kint_kernel (the
//      paper's dispatches): one warp per pair with the nodes spread over the
//      lanes (lb_kint.cuh).
// An FP64 call with one order for all pairs (v_stride 0) has its order's
// constants computed once per block (ScalarOrder).  FP64 calls of up to
// LB_SMALL_N pairs run lb_small_kernel alone, FP32 calls in tight mode
// lb_tiles32_kernel alone.
//
// The plain form computes in FP64; its exps and logs are evaluated in
// integer arithmetic where that is faster (lb_intmath.cuh).
#include <cuda_runtime.h>

#include <atomic>
#include <mutex>
#include <utility>
#include <vector>
#include <stdio.h>
#include <string.h>
#include <string>

#include "logbessel.h"
#include "lb_tile.cuh"
#include "lb_fastmath.cuh"

#define LB_VERSION "0.2.0"

using namespace lb;

namespace {

// Resident CTAs per SM the two kernels are built and launched for (launch
// bounds and persistent grid sizes: a multiple of the SM count).
// The tile kernel runs blocks of LB_TILE_THREADS threads, so a tile holds
// LB_TILE_THREADS * LB_ITEMS pairs: 2048 at 512 threads.  Larger tiles leave
// fewer partly filled 32-pair chunks at the end of each region's range of a
// tile (lanes that idle through an expression); at 512 threads and 3 CTAs
// per SM the SM keeps its 48 resident warps and 40 registers a thread, and
// the sweep's tile kernel time fell 4 % against 1024-pair tiles (256
// threads, 6 CTAs per SM).
#ifndef LB_TILE_THREADS
#define LB_TILE_THREADS 512
#endif
#ifndef LB_TILES_CTAS_PER_SM
#define LB_TILES_CTAS_PER_SM 3
#endif
#ifndef LB_KINT_CTAS_PER_SM
#define LB_KINT_CTAS_PER_SM 4
#endif
#ifndef LB_IN_TILE_THREADS_PER_SM
#define LB_IN_TILE_THREADS_PER_SM 768
#endif
#ifndef LB_LOW_THREADS
#define LB_LOW_THREADS 256
#endif
#ifndef LB_LOW_ITEMS
#define LB_LOW_ITEMS 1
#endif
#ifndef LB_MID_THREADS
#define LB_MID_THREADS 256
#endif
#ifndef LB_MID_ITEMS
#define LB_MID_ITEMS 2
#endif
#ifndef LB_SMALL_THREADS
#define LB_SMALL_THREADS 64
#endif
#ifndef LB_SMALL_N
#define LB_SMALL_N 2000
#endif
#ifndef LB_TILES32_CTAS_PER_SM
#define LB_TILES32_CTAS_PER_SM 6
#endif
#ifndef LB_KTRAP_THREADS
#define LB_KTRAP_THREADS 512
#endif
#ifndef LB_KTRAP_WINDOW
#define LB_KTRAP_WINDOW 15872
#endif
#ifndef LB_KTRAP_CTAS_PER_SM
#define LB_KTRAP_CTAS_PER_SM 3
#endif
#ifndef LB_KTRAP_CTAS_PER_SM_DX
#define LB_KTRAP_CTAS_PER_SM_DX 2
#endif
__host__ __device__ constexpr int ktrap_ctas(bool dx) { return dx ? LB_KTRAP_CTAS_PER_SM_DX : LB_KTRAP_CTAS_PER_SM; }

// K-integral queue entries: the pair's offset within its chunk (chunks hold
// at most 2^26 pairs) in the low 26 bits, the pair's class
// and band of work (8 kt_class + kt_band; FP64 tight, 0 otherwise) above them, so that a kernel
// that takes one class finds its pairs by reading the queue alone.
constexpr int kTileThreads = LB_TILE_THREADS;
constexpr int kTile = kTileThreads * LB_ITEMS;     // pairs per tile of the tile kernel
static_assert((1 << 26) % kTile == 0, "chunks of 2^26 pairs hold whole tiles");
constexpr int kQueueOffsetBits = 26;
constexpr uint32_t kQueueOffsetMask = (1u << kQueueOffsetBits) - 1u;

// Tile kernel: classify, bin per region in shared memory, evaluate the
// per-thread expressions (lb_tile.cuh); K fallback pairs go to a global queue
// for lb_ktrap_kernel (lb_kint_kernel in the paper's modes).  T = double
// (FP64) or float (FP32-mixed, the paper's modes).
// What bounds it: issue, spread over the pipes.  The mixed-order log K call
// at 6M pairs runs in 367 us (470 with the sums in FP64 and double-float),
// issue 66 % of cycles, FP64 pipe 48 %, ALU 47 %, integer multiplies 43 %,
// 1454 thread instructions per pair at 27 of 32 lanes, DRAM 4 %; the rest
// is waits at the tile's barriers and on fixed latencies, which more warps do
// not cover (registers allow 48 an SM).
// SO: one order for every argument (FP64 values, v_stride 0, no forced
// region): the order's constants once per block, and only the per-order
// forms of the expressions compiled in (each kernel carries one form's
// code, half the instruction footprint).
// NT: threads per block; the 2048-pair tiles of 512 threads suit calls that
// fill the GPU several times over, tiles of 512 pairs the smaller ones.
// KIN: the K fallback pairs are evaluated in the tile instead of queued.
// v == NULL: the order of every pair is v0 (v_stride 0).
// vmf_d >= 0: see tile_eval.
__host__ __device__ constexpr int tiles_ctas(int nt, bool kin) {
  return (kin ? LB_IN_TILE_THREADS_PER_SM : LB_TILES_CTAS_PER_SM * kTileThreads) / nt;
}
template <int KIND, bool DX, typename T, bool SO, int NT, int IT, bool KIN>
__global__ void __launch_bounds__(NT, tiles_ctas(NT, KIN))
lb_tiles_kernel(const T* __restrict__ v, int64_t v_stride, T v0, const T* __restrict__ x, T* __restrict__ out,
                int64_t n, int mode, int forced_region, unsigned int* __restrict__ qcount,
                uint32_t* __restrict__ queue, int64_t qcap, double vmf_d) {
  static_assert(!SO || (sizeof(T) == 8 && !DX), "per-order constants are built for FP64 values");
  constexpr int kPairs = NT * IT;
  __shared__ TileShared<T, NT, IT> S;
  const int tid = threadIdx.x;
  const int64_t ntiles = (n + kPairs - 1) / kPairs;
  if (v_stride == 0 && v) v0 = v[0];
  const unsigned long long* tab = nullptr;
  if constexpr (KIN) {
    __shared__ __align__(16) unsigned long long T2[2048];
    kt_load_table<NT>(T2);                          // a barrier of tile_bin stands between this and its use
    tab = T2;
  }
  const ScalarOrder* so = nullptr;
  if constexpr (SO) {
    __shared__ ScalarOrder SOC;
    scalar_order_setup<KIND, NT>(SOC, KIND == KIND_K ? fabs((double)v0) : (double)v0, mode);
    so = &SOC;
  }
  for (int64_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
    const int64_t t0 = tile * kPairs;
    tile_bin<KIND, DX, T, KIN>(S, v, v_stride, v0, x, t0, n, mode, forced_region);
    tile_eval<KIND, DX, T, SO, KIN>(S, out, t0, n, so, x, vmf_d, tab);
    if (KIND == KIND_K && sizeof(T) == 8 && !KIN) {
      const int c = S.rcount(R_FALLBACK), f0 = S.rbeg(R_FALLBACK);
      if (c > 0) {
        if (tid == 0) S.qbase = atomicAdd(qcount, (unsigned int)c);
        __syncthreads();
        const unsigned int b = S.qbase;
        for (int j = tid; j < c; j += NT) {
          const int li = S.list[f0 + j];
          uint32_t cl = 0;
          if constexpr (sizeof(T) == 8) {
            if (mode == MODE_TIGHT) {
              const double vi = S.sv[li], xi = S.sx[li];           // sv holds |v|
              const int c6 = kt_class(vi, xi, DX);
              cl = (uint32_t)(8 * c6 + kt_band(vi, xi, c6));
            }
          }
          // the pair's offset in the chunk (< 2^26) and its key above it
          if (LB_CHECK(b + j < qcap, 4u)) queue[b + j] = (uint32_t)(t0 + li) | (cl << kQueueOffsetBits);
        }
      }
    }
    __syncthreads();
  }
}

// Calls of few pairs: see warp_pair64.
template <int KIND, bool DX>
__global__ void __launch_bounds__(LB_SMALL_THREADS)
lb_small_kernel(const double* __restrict__ v, int64_t v_stride, double v0, const double* __restrict__ x,
                double* __restrict__ out, int64_t n, double vmf_d) {
  if (v_stride == 0 && v) v0 = v[0];
  const int64_t i = ((int64_t)blockIdx.x * LB_SMALL_THREADS + threadIdx.x) >> 5;
  __shared__ __align__(16) unsigned long long tab[KIND == KIND_K ? 2048 : 2];
  warp_pair64<KIND, DX, LB_SMALL_THREADS>(v, v_stride, v0, x, out, i, i < n, vmf_d, tab);
}

// K integral, tight FP64: one thread per queued pair (lb_ktrap.cuh).  A
// block takes windows of the queue, sorts each by the pairs' classes and
// bands in shared memory (a counting sort of 48 keys, two passes over the
// window) and hands out chunks of 32 pairs of one class to its warps,
// costliest class first, so that a warp runs one class's code on lanes that
// need about as many nodes.  The order of a key's pairs varies from run to
// run; a pair's result depends on the pair alone.
// What bounds it once the lanes are even is instruction fetch: the classes'
// code is larger than the instruction cache, so the warps of an SM should be
// in the same class.  Hence large blocks and windows of up to 15872 pairs (what
// 48 KB of shared memory hold beside the table), equal ones, as few per block
// as the queue needs: on the whole domain (6.9M queued pairs) 1.69 ms with
// 128-thread blocks and 1024-pair windows, 1.28 with 256 and 2048, 1.18 with
// 512 and 4096, 1.13 with 512 and 16384.  (The warp-per-pair Gauss rules it
// replaces took 19.1 ms on the same queue.)  There issue is at 60 %, the ALU
// at 56 %, integer multiplies at 47 %.
constexpr int kKtThreads = LB_KTRAP_THREADS;
constexpr int kKtWindow = LB_KTRAP_WINDOW;
static_assert(kKtWindow <= 65536, "16-bit offsets within a window");
template <bool DX>
__global__ void __launch_bounds__(kKtThreads, ktrap_ctas(DX))
lb_ktrap_kernel(const double* __restrict__ v, int64_t v_stride, const double* __restrict__ x,
                double* __restrict__ out, const unsigned int* __restrict__ qcount,
                const uint32_t* __restrict__ queue, int64_t n, int64_t qcap) {
  extern __shared__ __align__(16) unsigned char kt_shared[];
  unsigned long long* tab = reinterpret_cast<unsigned long long*>(kt_shared);
  uint16_t* list = reinterpret_cast<uint16_t*>(kt_shared + 2048 * sizeof(unsigned long long));
  __shared__ int count[64], beg[64], next_chunk;
  unsigned int cnt = *qcount;
  if (!LB_CHECK(cnt <= qcap, 8u)) cnt = (unsigned int)qcap;
  const int tid = threadIdx.x, lane = tid & 31;
  const int64_t share = ((int64_t)cnt + gridDim.x - 1) / gridDim.x;
  const int64_t rounds = (share + kKtWindow - 1) / kKtWindow;
  const int W = rounds ? (int)(((share + rounds - 1) / rounds + 31) & ~(int64_t)31) : 32;
  if ((int64_t)blockIdx.x * W >= (int64_t)cnt) return;     // the same for every thread of the block
  kt_load_table<kKtThreads>(tab);
  for (int64_t w0 = (int64_t)blockIdx.x * W; w0 < (int64_t)cnt; w0 += (int64_t)gridDim.x * W) {
    const int m = (int)min((int64_t)W, (int64_t)cnt - w0);
    if (tid < 64) count[tid] = 0;
    if (tid == 0) next_chunk = 0;
    __syncthreads();
    // pass 0 counts the keys, pass 1 places the entries; one atomic per key and warp
    for (int pass = 0; pass < 2; ++pass) {
      for (int j0 = tid - lane; j0 < m; j0 += kKtThreads) {
        const int j = j0 + lane;
        int key = -1;
        if (j < m) {
          const uint32_t e = queue[w0 + j];
          key = (int)(e >> kQueueOffsetBits);
          if (!LB_CHECK(key < 48, 32u)) key = 0;
          if (!LB_CHECK((int64_t)(e & kQueueOffsetMask) < n, 16u)) key = -1;
        }
        const unsigned peers = __match_any_sync(0xffffffffu, key);
        const int leader = __ffs(peers) - 1;
        int pos = 0;
        if (key >= 0 && lane == leader) pos = atomicAdd(pass ? &beg[key] : &count[key], __popc(peers));
        pos = __shfl_sync(0xffffffffu, pos, leader) + __popc(peers & ((1u << lane) - 1u));
        if (pass && key >= 0 && LB_CHECK(pos < kKtWindow, 1u)) list[pos] = (uint16_t)j;
      }
      __syncthreads();
      if (pass == 0) {
        if (tid < 32) {                            // exclusive prefix over the 64 key slots
          const int a = count[2 * lane], b = count[2 * lane + 1];
          int p = a + b;
#pragma unroll
          for (int o = 1; o < 32; o <<= 1) {
            const int u = __shfl_up_sync(0xffffffffu, p, o);
            if (lane >= o) p += u;
          }
          beg[2 * lane] = p - a - b;
          beg[2 * lane + 1] = p - b;
        }
        __syncthreads();
      }
    }
    // beg[k] is now the end of key k's entries
    for (;;) {
      int ch = 0;
      if (lane == 0) ch = atomicAdd(&next_chunk, 1);
      ch = __shfl_sync(0xffffffffu, ch, 0);
      // the chunk's class: chunks hold pairs of one class
      int c = 0, b = 0, e = 0;
#pragma unroll 1
      for (; c < 6; ++c) {
        b = c ? beg[8 * c - 1] : 0;
        e = beg[8 * c + 7];
        const int nc = (e - b + 31) >> 5;
        if (ch < nc) break;
        ch -= nc;
      }
      if (c == 6) break;
      const int j = b + (ch << 5) + lane;
      if (j < e) {
        const int64_t idx = (int64_t)(queue[w0 + list[j]] & kQueueOffsetMask);
        out[idx] = kt_eval<DX>(fabs(v[idx * v_stride]), x[idx], c, tab);
      }
      __syncwarp();
    }
    __syncthreads();
  }
}

// K integral of the paper's dispatches (Simpson's rule): one warp per queued
// pair, 32 pairs per warp batch, in queue order.
__global__ void __launch_bounds__(LB_THREADS, LB_KINT_CTAS_PER_SM)
lb_kint_kernel(const double* __restrict__ v, int64_t v_stride, const double* __restrict__ x,
               double* __restrict__ out, const unsigned int* __restrict__ qcount,
               const uint32_t* __restrict__ queue, int64_t n, int64_t qcap) {
  unsigned int cnt = *qcount;
  if (!LB_CHECK(cnt <= qcap, 8u)) cnt = (unsigned int)qcap;
  const int lane = threadIdx.x & 31;
  const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t b = warp * 32; b < (int64_t)cnt; b += nwarps * 32) {
    const int k = (int)min((int64_t)32, (int64_t)cnt - b);
    int64_t idx = (int64_t)(queue[b + (lane < k ? lane : 0)] & kQueueOffsetMask);
    const bool ok = LB_CHECK(idx < n, 16u);
    if (!ok) idx = 0;                              // clamped: the warp still runs the batch together
    const double val = kint_warp_batch(fabs(v[idx * v_stride]), x[idx], k, lane);
    if (lane < k && ok) out[idx] = val;
  }
}

// FP32, tight mode: see warp_pairs32.  Bound by issue: log I over mixed
// orders, 24M pairs, 128 us (387 with the binned tiles), 155 thread
// instructions per pair, issue 74 %, ALU 51 %, DRAM 17 % at 6M pairs; log K
// over the whole domain, 16M pairs, 195 us (2670 with a warp per integral; 217,
// issue 69 % and waits for instructions, with the edges' code in the loop
// instead of called), issue 75 %.
template <int KIND, int VEC>
__global__ void __launch_bounds__(LB_THREADS, LB_TILES32_CTAS_PER_SM)
lb_tiles32_kernel(const float* __restrict__ v, int64_t v_stride, const float* __restrict__ x,
                  float* __restrict__ out, int64_t n) {
  __shared__ Warp32 W[LB_THREADS / 32];
  const int warps = blockDim.x >> 5, w = threadIdx.x >> 5;
  warp_pairs32<KIND, VEC>(W[w], v, v_stride, x, out, 0, n, (int64_t)w * gridDim.x + blockIdx.x,
                          (int64_t)warps * gridDim.x);
}

template <int KIND>
__global__ void lb_classify_kernel32(const float* __restrict__ v, int64_t v_stride,
                                     const float* __restrict__ x, uint8_t* __restrict__ reg,
                                     int64_t n, int mode) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    float vi = v[i * v_stride];
    const float xi = x[i];
    if (KIND == KIND_K) vi = fabsf(vi);
    float sp;
    reg[i] = special_value32<KIND>(vi, xi, &sp) ? (uint8_t)R_SPECIAL : (uint8_t)classify32(vi, xi, mode, KIND == KIND_K ? WIDE_K : WIDE_I);
  }
}

template <int KIND>
__global__ void lb_classify_kernel(const double* __restrict__ v, int64_t v_stride,
                                   const double* __restrict__ x, uint8_t* __restrict__ reg,
                                   int64_t n, int mode) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    double vi = v[i * v_stride];
    const double xi = x[i];
    if (KIND == KIND_K) vi = fabs(vi);
    double sp;
    reg[i] = special_value<KIND>(vi, xi, &sp) ? (uint8_t)R_SPECIAL : (uint8_t)classify(vi, xi, mode, KIND == KIND_K ? WIDE_K : WIDE_I);
  }
}

// Elementwise exp/log for checking the table-driven implementations against
// the libm ones: which = 0 fm_exp, 1 fm_log, 2 exp, 3 log; and CUDA's
// special-purpose Bessel functions of orders 0 and 1 (the comparison system
// of paper Sec. 6.1): 4 log(cyl_bessel_i0), 5 log(cyl_bessel_i1).
__global__ void lb_math_kernel(int which, const double* __restrict__ in, double* __restrict__ out, int64_t n) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const double a = in[i];
    double r;
    switch (which) {
      case 0: r = fm_exp(a); break;
      case 1: r = fm_log(a); break;
      case 2: r = exp(a); break;
      case 3: r = log(a); break;
      case 4: r = log(cyl_bessel_i0(a)); break;
      case 5: r = log(cyl_bessel_i1(a)); break;
      case 6: r = fm_exp_term(a); break;
      case 7: r = ix_exp(a); break;
      case 8: r = ix_log(a); break;
      case 9: r = ix_rcp(a); break;
      case 10: r = ix_rsqrt(a); break;
      case 11: r = __longlong_as_double(ix_log_q53(a)); break;          // the Q53 integer's bits
      default: r = __longlong_as_double((long long)ix_exp_q58_fx(__double_as_longlong(a))); break;
    }
    out[i] = r;
  }
}

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------
thread_local std::string g_last_error;

lb_status fail(lb_status st, const char* fmt, const char* a = "", long long b = 0) {
  char buf[512];
  snprintf(buf, sizeof buf, fmt, a, b);
  g_last_error = buf;
  return st;
}

lb_status check_launch(const char* what) {
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) {
    g_last_error = std::string(what) + ": " + cudaGetErrorString(e);
    return LB_ECUDA;
  }
  return LB_OK;
}

int sm_count() {
  static std::mutex mu;
  static int cache[64] = {0};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 152;
  std::lock_guard<std::mutex> lk(mu);
  if (cache[dev] == 0) {
    int sms = 0;
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms <= 0) sms = 152;
    cache[dev] = sms;
  }
  return cache[dev];
}

// ---------------------------------------------------------------------------
// launch accounting and optional per-kernel CUDA-event timing
// ---------------------------------------------------------------------------
enum ProfSlotId { PS_TILES = 0, PS_KINT = 1, PS_CLASSIFY = 2, PS_AUX = 3, PS_NSLOTS = 4 };
const char* const kSlotNames[PS_NSLOTS] = {"lb_tiles_kernel", "lb_kint_kernel", "lb_classify_kernel",
                                           "lb_aux_kernels"};

struct ProfState {
  std::mutex mu;
  bool on = false;
  long long launches[PS_NSLOTS] = {0, 0, 0, 0};
  long long timed[PS_NSLOTS] = {0, 0, 0, 0};
  double ms[PS_NSLOTS] = {0, 0, 0, 0};
  std::vector<std::pair<int, std::pair<cudaEvent_t, cudaEvent_t>>> pending;
};
ProfState& prof() {
  static ProfState p;
  return p;
}
std::atomic<long long> g_total_launches{0};

void prof_drain_locked(ProfState& P) {
  for (auto& e : P.pending) {
    float t = 0.f;
    if (cudaEventSynchronize(e.second.second) == cudaSuccess &&
        cudaEventElapsedTime(&t, e.second.first, e.second.second) == cudaSuccess) {
      P.ms[e.first] += t;
      P.timed[e.first] += 1;
    }
    cudaEventDestroy(e.second.first);
    cudaEventDestroy(e.second.second);
  }
  P.pending.clear();
}

// Launch `body` (one kernel launch) on stream st under slot `slot`.
template <typename F>
lb_status launch(int slot, cudaStream_t st, F&& body) {
  ProfState& P = prof();
  cudaEvent_t a = nullptr, b = nullptr;
  bool timed = false;
  {
    std::lock_guard<std::mutex> lk(P.mu);
    timed = P.on;
  }
  if (timed && (cudaEventCreate(&a) != cudaSuccess || cudaEventCreate(&b) != cudaSuccess)) timed = false;
  if (timed) cudaEventRecord(a, st);
  body();
  lb_status s = check_launch(kSlotNames[slot]);
  g_total_launches.fetch_add(1);
  {
    std::lock_guard<std::mutex> lk(P.mu);
    P.launches[slot] += 1;
    if (timed) {
      cudaEventRecord(b, st);
      P.pending.push_back({slot, {a, b}});
    }
  }
  return s;
}

lb_status validate(lb_dtype dtype, const void* v, int64_t v_stride, const void* x, const void* out,
                   int64_t n, int mode) {
  if (n < 0) return fail(LB_EINVAL, "n must be >= 0 (got %s%lld)", "", (long long)n);
  if (dtype != LB_F64 && dtype != LB_F32) return fail(LB_EINVAL, "unknown dtype %s%lld", "", (long long)dtype);
  if (mode < 0 || mode > 2) return fail(LB_EINVAL, "unknown mode %s%lld", "", (long long)mode);
  if (v_stride != 0 && v_stride != 1) return fail(LB_EINVAL, "v_stride must be 0 or 1 (got %s%lld)", "", (long long)v_stride);
  if (n > 0 && (!v || !x || !out)) return fail(LB_EINVAL, "NULL %s pointer with n = %lld", !v ? "v" : (!x ? "x" : "out"), (long long)n);
  return LB_OK;
}

// Largest chunk handled with one queue: the queue entries hold 26-bit offsets.
const int64_t kChunk = (int64_t)1 << kQueueOffsetBits;
// Smallest caller workspace: the counters and the queue of one tile.
const int64_t kWsMin = 256 + 4 * kTile;
static_assert(256 + 4 * kTile == 8448, "the documented smallest workspace");

// FP32, tight mode.  16-byte loads when the pointers allow them and there are
// enough pairs for every SM's resident warps; otherwise one pair per lane,
// and slices dealt to the blocks in turn, so that a small call uses as many
// SMs as it can.  2^31 pairs per launch (32-bit offsets in the lists).
template <int KIND>
lb_status run_tiles32(const float* v, int64_t v_stride, const float* x, float* out, int64_t n, cudaStream_t st) {
  const int64_t most = (int64_t)sm_count() * LB_TILES32_CTAS_PER_SM;
  const uintptr_t al = (uintptr_t)x | (uintptr_t)out | (v_stride ? (uintptr_t)v : 0);
  const bool wide = (al & 15) == 0 && n > most * LB_THREADS;
  lb_status s = LB_OK;
  for (int64_t c0 = 0; c0 < n && s == LB_OK; c0 += (int64_t)1 << 31) {
    const int64_t cn = n - c0 < ((int64_t)1 << 31) ? n - c0 : (int64_t)1 << 31;
    const int64_t slices = (cn + (wide ? 127 : 31)) / (wide ? 128 : 32);
    const int grid = (int)(slices < most ? slices : most);
    const int64_t per = (slices + grid - 1) / grid;        // warps a block can use
    const int threads = (int)(per < LB_THREADS / 32 ? per : LB_THREADS / 32) * 32;
    s = launch(PS_TILES, st, [&] {
      if (wide) lb_tiles32_kernel<KIND, 4><<<grid, threads, 0, st>>>(v + c0 * v_stride, v_stride, x + c0, out + c0, cn);
      else lb_tiles32_kernel<KIND, 1><<<grid, threads, 0, st>>>(v + c0 * v_stride, v_stride, x + c0, out + c0, cn);
    });
  }
  return s;
}

// Enqueue the evaluation of n pairs.  The FP64 K fallback goes through a queue
// of 32-bit pair offsets in scratch memory (qcount: the counter, queue:
// min(n, chunk) entries), processed chunk by chunk; `scratch` supplies it,
// or, when NULL, it comes from the stream-ordered allocator.
//
// FP64 calls of total_n pairs (the caller's n; passes and pieces of one call
// take the same route, so that their results are those of one pass):
//   up to LB_SMALL_N  lb_small_kernel alone (tight mode);
//   below 2^17        tiles of 256 pairs, one per thread, the K fallback in the
//                     tile (tight mode): one launch and no scratch;
//   below 2^20        tiles of 512 pairs, two per thread, K fallback queued
//                     (see large_tiles for what leaves them sooner);
//   from there        tiles of 2048 pairs, four per thread, K fallback queued.
// Device time of a call on the mixed-order sweep, log I / log K, us: 1000
// pairs 12 / 12 (small kernel) against 16 / 15 (256-pair tiles); 4000 pairs 17
// / 16 (256-pair tiles) against 19 / 21 (small kernel); 24000 pairs 17 / 17
// against 25 / 33 (small kernel), 19 / 36 (512-pair tiles, queued) and 32 / 49
// (2048-pair tiles); 100000 pairs 22 / 27 against 23 / 43 and 33 / 53; 200000
// pairs 27 / 49 against 33 / 55 (2048-pair tiles); 1M pairs 91 / 108 against 86
// / 110, log C_2048 72 against 79.
constexpr int64_t kMidInTile = (int64_t)1 << 17, kMid = (int64_t)1 << 20;

template <int KIND, bool DX, typename T, bool SO, int NT, int IT, bool KIN>
lb_status launch_tiles(int sms, cudaStream_t st, const T* v, int64_t v_stride, T v0, const T* x, T* out, int64_t n,
                       int mode, int forced_region, unsigned int* qcount, uint32_t* queue, int64_t cap, double vmf_d) {
  const int64_t ntiles = (n + NT * IT - 1) / (NT * IT), most = (int64_t)sms * tiles_ctas(NT, KIN);
  const int grid = (int)(ntiles < most ? ntiles : most);
  return launch(PS_TILES, st, [&] {
    lb_tiles_kernel<KIND, DX, T, SO, NT, IT, KIN><<<grid, NT, 0, st>>>(v, v_stride, v0, x, out, n, mode, forced_region,
                                                                  qcount, queue, cap, vmf_d);
  });
}

// Whether a call of n pairs between 2^17 and 2^20 leaves the 512-pair tiles: one
// wave of them holds 467000 pairs on 152 SMs, one of 2048-pair tiles 934000.  In
// between, the small ones run a second wave that is partly empty (a quarter of
// one is made up for by the emptier SMs it runs on).  The large ones take it
// there for log I's derivative (600000 pairs, order 1/2: 83 us with the small
// ones, 71 with the large; order 4 85 / 70, mixed sweep 75 / 64; 500000 pairs of
// U_K 37 / 43) and for the paper's dispatches (whole domain, 600000 pairs, log I
// 155 / 136, its derivative 176 / 150; order 4, 500000 pairs 106 / 118, 1M 193 /
// 216).  (The tight values' kernels and log K's derivative are as fast either
// way.)
inline bool large_tiles(int sms, int mode, bool dx_i, int64_t n) {
  constexpr int64_t kMidWave = tiles_ctas(LB_MID_THREADS, false) * LB_MID_THREADS * LB_MID_ITEMS;
  return (mode != MODE_TIGHT || dx_i) && n > sms * kMidWave / 4 * 5 &&
         n <= (int64_t)sms * LB_TILES_CTAS_PER_SM * kTile;
}

// The tile kernel of a pass of n pairs: one order per call has its constants
// computed per block, where there are enough pairs to pay for that.
template <int KIND, bool DX, typename T>
lb_status run_tiles(int sms, cudaStream_t st, const T* v, int64_t v_stride, T v0, const T* x, T* out, int64_t n,
                    int mode, int forced_region, unsigned int* qcount, uint32_t* queue, int64_t cap, int64_t total_n,
                    double vmf_d) {
  if constexpr (sizeof(T) == 8) {
    // (an order known here to be past 16 -- the vMF form's d/2 - 1 usually is --
    // takes the general kernel: U_4 sums are short, and the one-order kernel's
    // set-up pays in large calls only.  log C_2048: 600000 values 54 us against
    // 58, 1M 78 against 81, 4M 258 against 246)
    const bool so = !DX && v_stride == 0 && forced_region < 0 && (v || (double)v0 <= 16.0);
    if (total_n < kMid && forced_region < 0 && !large_tiles(sms, mode, KIND == KIND_I && DX && v, total_n)) {
      if (so && total_n >= kMidInTile)
        return launch_tiles<KIND, DX, T, !DX, LB_MID_THREADS, LB_MID_ITEMS, false>(sms, st, v, v_stride, v0, x, out, n, mode,
                                                                  forced_region, qcount, queue, cap, vmf_d);
      if (total_n < kMidInTile)
        return launch_tiles<KIND, DX, T, false, LB_LOW_THREADS, LB_LOW_ITEMS, false>(
            sms, st, v, v_stride, v0, x, out, n, mode, forced_region, qcount, queue, cap, vmf_d);
      return launch_tiles<KIND, DX, T, false, LB_MID_THREADS, LB_MID_ITEMS, false>(
          sms, st, v, v_stride, v0, x, out, n, mode, forced_region, qcount, queue, cap, vmf_d);
    }
    if (so)
      return launch_tiles<KIND, DX, T, !DX, kTileThreads, LB_ITEMS, false>(sms, st, v, v_stride, v0, x, out, n, mode,
                                                                 forced_region, qcount, queue, cap, vmf_d);
  }
  return launch_tiles<KIND, DX, T, false, kTileThreads, LB_ITEMS, false>(sms, st, v, v_stride, v0, x, out, n, mode,
                                                               forced_region, qcount, queue, cap, vmf_d);
}

template <int KIND, bool DX, typename T>
lb_status run_impl(const T* v, int64_t v_stride, const T* x, T* out, int64_t n, int mode, int forced_region,
                   cudaStream_t st, void* scratch, int64_t chunk, int64_t total_n, T v0 = T(0), double vmf_d = -1.0) {
  const int sms = sm_count();
  if (KIND == KIND_K && sizeof(T) == 4 && mode != MODE_TIGHT && (forced_region < 0 || forced_region == R_FALLBACK))
    return fail(LB_ENOTSUP, "%sthe FP32 K integral is implemented for LB_TIGHT only", "", 0);
  if constexpr (sizeof(T) == 4) {
    if (mode == MODE_TIGHT && forced_region < 0) return run_tiles32<KIND>(v, v_stride, x, out, n, st);
  } else if (mode == MODE_TIGHT && forced_region < 0) {
    if (total_n <= LB_SMALL_N) {
      const int grid = (int)((n * 32 + LB_SMALL_THREADS - 1) / LB_SMALL_THREADS);   // a warp per pair
      return launch(PS_TILES, st, [&] {
        lb_small_kernel<KIND, DX><<<grid, LB_SMALL_THREADS, 0, st>>>(v, v_stride, v0, x, out, n, vmf_d);
      });
    }
    if (KIND == KIND_K && total_n < kMidInTile)
      return launch_tiles<KIND, DX, T, false, LB_LOW_THREADS, LB_LOW_ITEMS, KIND == KIND_K>(sms, st, v, v_stride, v0, x, out, n, mode,
                                                                           forced_region, nullptr, nullptr, 0, vmf_d);
  }
  if (KIND == KIND_I || sizeof(T) == 4 || (forced_region >= 0 && forced_region != R_FALLBACK))
    return run_tiles<KIND, DX, T>(sms, st, v, v_stride, v0, x, out, n, mode, forced_region, nullptr, nullptr, 0,
                                  total_n, vmf_d);
  if constexpr (sizeof(T) == 8) {
    // queue entries a pass can write: every workspace holds at least this many
    const int64_t cap = n < chunk ? n : chunk;
    void* ws = scratch;
    if (!ws) {
      const size_t bytes = 256 + (size_t)cap * sizeof(uint32_t);
      if (cudaMallocAsync(&ws, bytes, st) != cudaSuccess) {
        cudaGetLastError();
        return fail(LB_ENOMEM, "cudaMallocAsync of %s%lld bytes failed", "", (long long)bytes);
      }
    }
    unsigned int* qcount = (unsigned int*)ws;
    uint32_t* queue = (uint32_t*)((char*)ws + 256);
    lb_status status = LB_OK;
    for (int64_t c0 = 0; c0 < n && status == LB_OK; c0 += chunk) {
      const int64_t cn = (n - c0) < chunk ? (n - c0) : chunk;
      if (cudaMemsetAsync(qcount, 0, sizeof(unsigned int), st) != cudaSuccess) { status = check_launch("cudaMemsetAsync"); break; }
      const T* vc = v + c0 * v_stride;
      const T* xc = x + c0;
      T* oc = out + c0;
      status = run_tiles<KIND, DX, T>(sms, st, vc, v_stride, v0, xc, oc, cn, mode, forced_region, qcount, queue, cap,
                                      total_n, vmf_d);
      if (status != LB_OK) break;
      if (mode == MODE_TIGHT) {
        // the queue's length is on the device: a block per 32 pairs it can hold, at most the resident ones
        const int64_t want = (cn + 31) / 32, most = (int64_t)sms * ktrap_ctas(DX);
        const int kgrid = (int)(want < most ? want : most);
        constexpr int kShared = 2048 * 8 + 2 * kKtWindow;   // with the static arrays below 48 KB: no opt-in
        status = launch(PS_KINT, st, [&] {
          lb_ktrap_kernel<DX><<<kgrid, kKtThreads, kShared, st>>>(vc, v_stride, xc, oc, qcount, queue, cn, cap);
        });
      } else {
        const int kgrid = sms * 2 * LB_KINT_CTAS_PER_SM;
        status = launch(PS_KINT, st, [&] {
          lb_kint_kernel<<<kgrid, LB_THREADS, 0, st>>>(vc, v_stride, xc, oc, qcount, queue, cn, cap);
        });
      }
    }
    if (!scratch) cudaFreeAsync(ws, st);
    return status;
  }
  return LB_OK;
}

template <int KIND, bool DX>
lb_status run(const double* v, int64_t v_stride, const double* x, double* out, int64_t n, int mode,
              int forced_region, cudaStream_t st) {
  return run_impl<KIND, DX, double>(v, v_stride, x, out, n, mode, forced_region, st, nullptr, kChunk, n);
}

lb_status run32(int kind, const float* v, int64_t v_stride, const float* x, float* out, int64_t n, int mode,
                int forced_region, cudaStream_t st) {
  if (kind == KIND_I) return run_impl<KIND_I, false, float>(v, v_stride, x, out, n, mode, forced_region, st, nullptr, kChunk, n);
  return run_impl<KIND_K, false, float>(v, v_stride, x, out, n, mode, forced_region, st, nullptr, kChunk, n);
}

// Fixed scratch for logbessel_k_noalloc: the queue counter (first 256
// bytes) and the queue of the K fallback pairs, for at most
// LB_NOALLOC_MAX_PAIRS pairs per call.  It lives in the module's global
// memory for as long as the library is loaded, on every device that loads it.
#define LB_NOALLOC_MAX_PAIRS (1 << 20)
static __device__ __align__(256) uint32_t lb_noalloc_scratch[64 + LB_NOALLOC_MAX_PAIRS];

// Device address of lb_noalloc_scratch in the current context, looked up on
// every call: cudaGetSymbolAddress allocates nothing, and a cached address
// would go stale when the device's primary context is torn down and made
// again (cudaDeviceReset), since the module then reloads elsewhere.
void* noalloc_scratch_address() {
  void* p = nullptr;
  const cudaError_t e = cudaGetSymbolAddress(&p, lb_noalloc_scratch);
  if (e != cudaSuccess) {
    cudaGetLastError();
    g_last_error = std::string("logbessel_k_noalloc: cudaGetSymbolAddress failed: ") + cudaGetErrorString(e);
    return nullptr;
  }
  return p;
}

}  // namespace

extern "C" {

lb_status logbessel_i(lb_dtype dtype, const void* v, int64_t v_stride, const void* x, void* out,
                      int64_t n, lb_mode mode, void* cuda_stream) {
  lb_status s = validate(dtype, v, v_stride, x, out, n, (int)mode);
  if (s != LB_OK || n == 0) return s;
  if (dtype == LB_F32)
    return run32(KIND_I, (const float*)v, v_stride, (const float*)x, (float*)out, n, (int)mode, -1,
                 (cudaStream_t)cuda_stream);
  return run<KIND_I, false>((const double*)v, v_stride, (const double*)x, (double*)out, n, (int)mode, -1,
                            (cudaStream_t)cuda_stream);
}

lb_status logbessel_k(lb_dtype dtype, const void* v, int64_t v_stride, const void* x, void* out,
                      int64_t n, lb_mode mode, void* cuda_stream) {
  lb_status s = validate(dtype, v, v_stride, x, out, n, (int)mode);
  if (s != LB_OK || n == 0) return s;
  if (dtype == LB_F32)
    return run32(KIND_K, (const float*)v, v_stride, (const float*)x, (float*)out, n, (int)mode, -1,
                 (cudaStream_t)cuda_stream);
  return run<KIND_K, false>((const double*)v, v_stride, (const double*)x, (double*)out, n, (int)mode, -1,
                            (cudaStream_t)cuda_stream);
}

lb_status logbessel_i_dx(lb_dtype dtype, const void* v, int64_t v_stride, const void* x, void* out,
                         int64_t n, lb_mode mode, void* cuda_stream) {
  lb_status s = validate(dtype, v, v_stride, x, out, n, (int)mode);
  if (s != LB_OK || n == 0) return s;
  if (dtype != LB_F64) return fail(LB_ENOTSUP, "%sthe derivatives are implemented for LB_F64 only", "", 0);
  return run<KIND_I, true>((const double*)v, v_stride, (const double*)x, (double*)out, n, (int)mode, -1,
                           (cudaStream_t)cuda_stream);
}

lb_status logbessel_k_dx(lb_dtype dtype, const void* v, int64_t v_stride, const void* x, void* out,
                         int64_t n, lb_mode mode, void* cuda_stream) {
  lb_status s = validate(dtype, v, v_stride, x, out, n, (int)mode);
  if (s != LB_OK || n == 0) return s;
  if (dtype != LB_F64) return fail(LB_ENOTSUP, "%sthe derivatives are implemented for LB_F64 only", "", 0);
  if (mode != LB_TIGHT) return fail(LB_ENOTSUP, "%sd/dx log K is implemented for LB_TIGHT only", "", 0);
  return run<KIND_K, true>((const double*)v, v_stride, (const double*)x, (double*)out, n, (int)mode, -1,
                           (cudaStream_t)cuda_stream);
}

lb_status logbessel_k_noalloc(lb_dtype dtype, const void* v, int64_t v_stride, const void* x, void* out,
                              int64_t n, lb_mode mode, void* cuda_stream) {
  lb_status s = validate(dtype, v, v_stride, x, out, n, (int)mode);
  if (s != LB_OK || n == 0) return s;
  if (dtype != LB_F64) return fail(LB_ENOTSUP, "%slogbessel_k_noalloc supports LB_F64 only", "", 0);
  if (n > LB_NOALLOC_MAX_PAIRS)
    return fail(LB_EINVAL, "%slogbessel_k_noalloc takes at most 1048576 pairs per call (got %lld)", "", (long long)n);
  void* scratch = noalloc_scratch_address();
  if (!scratch) return LB_ECUDA;
  return run_impl<KIND_K, false, double>((const double*)v, v_stride, (const double*)x, (double*)out, n, (int)mode,
                                         -1, (cudaStream_t)cuda_stream, scratch, LB_NOALLOC_MAX_PAIRS, n);
}

int64_t logbessel_workspace_bytes(int64_t n) {
  if (n < 0) return 0;
  const int64_t m = (n + kTile - 1) / kTile * kTile;        // passes hold whole tiles
  return 256 + 4 * (m < kTile ? kTile : (m < kChunk ? m : kChunk));
}

lb_status logbessel_k_ws(lb_dtype dtype, const void* v, int64_t v_stride, const void* x, void* out, int64_t n,
                         lb_mode mode, void* workspace, int64_t ws_bytes, void* cuda_stream) {
  lb_status s = validate(dtype, v, v_stride, x, out, n, (int)mode);
  if (s != LB_OK) return s;
  if (!workspace || ((uintptr_t)workspace & 255) || ws_bytes < kWsMin)
    return fail(LB_EINVAL, "%sworkspace must be non-NULL, 256-byte aligned and at least 8448 bytes (got %lld)", "",
                (long long)ws_bytes);
  if (n == 0) return LB_OK;
  // passes start on tile boundaries, so the results equal those of one pass
  const int64_t cap0 = (ws_bytes - 256) / 4;
  const int64_t cap = ((cap0 < kChunk ? cap0 : kChunk) / kTile) * kTile;
  cudaStream_t st = (cudaStream_t)cuda_stream;
  if (dtype == LB_F32)
    return run_impl<KIND_K, false, float>((const float*)v, v_stride, (const float*)x, (float*)out, n, (int)mode, -1,
                                          st, workspace, cap, n);
  return run_impl<KIND_K, false, double>((const double*)v, v_stride, (const double*)x, (double*)out, n, (int)mode,
                                         -1, st, workspace, cap, n);
}

lb_status logbessel_k_dx_ws(lb_dtype dtype, const void* v, int64_t v_stride, const void* x, void* out, int64_t n,
                            lb_mode mode, void* workspace, int64_t ws_bytes, void* cuda_stream) {
  lb_status s = validate(dtype, v, v_stride, x, out, n, (int)mode);
  if (s != LB_OK) return s;
  if (!workspace || ((uintptr_t)workspace & 255) || ws_bytes < kWsMin)
    return fail(LB_EINVAL, "%sworkspace must be non-NULL, 256-byte aligned and at least 8448 bytes (got %lld)", "",
                (long long)ws_bytes);
  if (n == 0) return LB_OK;
  if (dtype != LB_F64) return fail(LB_ENOTSUP, "%sthe derivatives are implemented for LB_F64 only", "", 0);
  if (mode != LB_TIGHT) return fail(LB_ENOTSUP, "%sd/dx log K is implemented for LB_TIGHT only", "", 0);
  // passes start on tile boundaries, so the results equal those of one pass
  const int64_t cap0 = (ws_bytes - 256) / 4;
  const int64_t cap = ((cap0 < kChunk ? cap0 : kChunk) / kTile) * kTile;
  return run_impl<KIND_K, true, double>((const double*)v, v_stride, (const double*)x, (double*)out, n, (int)mode, -1,
                                        (cudaStream_t)cuda_stream, workspace, cap, n);
}

lb_status logbessel_classify(int kind, lb_dtype dtype, const void* v, int64_t v_stride,
                             const void* x, uint8_t* region_out, int64_t n, lb_mode mode,
                             void* cuda_stream) {
  if (kind != 0 && kind != 1) return fail(LB_EINVAL, "kind must be 0 (I) or 1 (K), got %s%lld", "", (long long)kind);
  lb_status s = validate(dtype, v, v_stride, x, region_out, n, (int)mode);
  if (s != LB_OK || n == 0) return s;
  const int grid = sm_count() * 4;
  cudaStream_t st = (cudaStream_t)cuda_stream;
  if (dtype == LB_F32)
    return launch(PS_CLASSIFY, st, [&] {
      if (kind == 0)
        lb_classify_kernel32<KIND_I><<<grid, LB_THREADS, 0, st>>>((const float*)v, v_stride, (const float*)x, region_out, n, (int)mode);
      else
        lb_classify_kernel32<KIND_K><<<grid, LB_THREADS, 0, st>>>((const float*)v, v_stride, (const float*)x, region_out, n, (int)mode);
    });
  return launch(PS_CLASSIFY, st, [&] {
    if (kind == 0)
      lb_classify_kernel<KIND_I><<<grid, LB_THREADS, 0, st>>>((const double*)v, v_stride, (const double*)x, region_out, n, (int)mode);
    else
      lb_classify_kernel<KIND_K><<<grid, LB_THREADS, 0, st>>>((const double*)v, v_stride, (const double*)x, region_out, n, (int)mode);
  });
}

lb_status logbessel_eval_region(int kind, lb_dtype dtype, const void* v, int64_t v_stride,
                                const void* x, void* out, int64_t n, int region, lb_mode mode,
                                void* cuda_stream) {
  if (kind != 0 && kind != 1) return fail(LB_EINVAL, "kind must be 0 (I) or 1 (K), got %s%lld", "", (long long)kind);
  if (region < 0 || region > R_U9 || region == R_SPECIAL)
    return fail(LB_EINVAL, "region %s%lld is not an expression", "", (long long)region);
  lb_status s = validate(dtype, v, v_stride, x, out, n, (int)mode);
  if (s != LB_OK || n == 0) return s;
  cudaStream_t st = (cudaStream_t)cuda_stream;
  if (dtype == LB_F32)
    return run32(kind, (const float*)v, v_stride, (const float*)x, (float*)out, n, (int)mode, region, st);
  if (kind == 0)
    return run<KIND_I, false>((const double*)v, v_stride, (const double*)x, (double*)out, n, (int)mode, region, st);
  return run<KIND_K, false>((const double*)v, v_stride, (const double*)x, (double*)out, n, (int)mode, region, st);
}

lb_status logbessel_vmf_log_c(lb_dtype dtype, double d, const void* kappa, void* out, int64_t n, int deriv,
                              void* cuda_stream) {
  if (!(d >= 2.0) || !isfinite(d)) return fail(LB_EINVAL, "dimension d must be finite and >= 2 (got %s%lld)", "", (long long)d);
  if (deriv != 0 && deriv != 1) return fail(LB_EINVAL, "deriv must be 0 or 1 (got %s%lld)", "", (long long)deriv);
  lb_status s = validate(dtype, kappa, 0, kappa, out, n, 0);
  if (s != LB_OK || n == 0) return s;
  if (dtype != LB_F64) return fail(LB_ENOTSUP, "%sthe vMF log-normaliser is implemented for LB_F64 only", "", 0);
  cudaStream_t st = (cudaStream_t)cuda_stream;
  const double nu = 0.5 * d - 1.0, *k = (const double*)kappa;
  if (deriv)
    return run_impl<KIND_I, true, double>(nullptr, 0, k, (double*)out, n, MODE_TIGHT, -1, st, nullptr, kChunk, n, nu, d);
  return run_impl<KIND_I, false, double>(nullptr, 0, k, (double*)out, n, MODE_TIGHT, -1, st, nullptr, kChunk, n, nu, d);
}

lb_status logbessel_math_eval(int which, const double* in, double* out, int64_t n, void* cuda_stream) {
  if (which < 0 || which > 12) return fail(LB_EINVAL, "which must be 0..12 (got %s%lld)", "", (long long)which);
  if (n < 0 || (n > 0 && (!in || !out))) return fail(LB_EINVAL, "bad buffer or size %s%lld", "", (long long)n);
  if (n == 0) return LB_OK;
  cudaStream_t st = (cudaStream_t)cuda_stream;
  const int grid = sm_count() * 4;
  return launch(PS_AUX, st, [&] { lb_math_kernel<<<grid, LB_THREADS, 0, st>>>(which, in, out, n); });
}

// Chunk slots of the pipeline: one more than the three stages, so that a
// copy that stalls for a while (the host memory is shared) does not stop
// the evaluation of the next chunk.
constexpr int kHostSlots = 4;

// Streams, events and the device buffer of logbessel_host, kept per device
// from one call to the next: allocating and releasing the few hundred MB of
// chunk buffers on every call (the stream-ordered pool returns them to the
// driver at each synchronization) costs more than a short call's evaluation.
// A call holds its device's lock from start to end.
struct HostPipe {
  std::mutex mu;
  bool init = false;
  cudaStream_t st[4] = {};                      // copy-in, compute (even pieces), copy-out, compute (odd)
  cudaEvent_t ev_in[kHostSlots] = {}, ev_comp[kHostSlots] = {}, ev_out[kHostSlots] = {};
  char* dbuf = nullptr;
  size_t bytes = 0;
};
constexpr int kMaxDevices = 64;

HostPipe& host_pipe(int dev) {
  static HostPipe pipes[kMaxDevices];
  return pipes[dev];
}

void host_pipe_destroy(HostPipe& P) {
  if (P.dbuf) cudaFree(P.dbuf);
  for (int i = 0; i < kHostSlots; ++i) {
    if (P.ev_in[i]) cudaEventDestroy(P.ev_in[i]);
    if (P.ev_comp[i]) cudaEventDestroy(P.ev_comp[i]);
    if (P.ev_out[i]) cudaEventDestroy(P.ev_out[i]);
    P.ev_in[i] = P.ev_comp[i] = P.ev_out[i] = nullptr;
  }
  for (int i = 0; i < 4; ++i) {
    if (P.st[i]) cudaStreamDestroy(P.st[i]);
    P.st[i] = nullptr;
  }
  P.dbuf = nullptr;
  P.bytes = 0;
  P.init = false;
}

bool host_pipe_init(HostPipe& P) {
  bool ok = true;
  for (int i = 0; i < 4 && ok; ++i) ok = cudaStreamCreateWithFlags(&P.st[i], cudaStreamNonBlocking) == cudaSuccess;
  for (int i = 0; i < kHostSlots && ok; ++i)
    ok = cudaEventCreateWithFlags(&P.ev_in[i], cudaEventDisableTiming) == cudaSuccess &&
         cudaEventCreateWithFlags(&P.ev_comp[i], cudaEventDisableTiming) == cudaSuccess &&
         cudaEventCreateWithFlags(&P.ev_out[i], cudaEventDisableTiming) == cudaSuccess;
  if (!ok) {
    cudaGetLastError();
    host_pipe_destroy(P);
    return false;
  }
  P.init = true;
  return true;
}

lb_status logbessel_host(int fn, lb_dtype dtype, const void* v, int64_t v_stride, const void* x, void* out,
                         int64_t n, lb_mode mode, int64_t chunk) {
  if (fn < 0 || fn > 3) return fail(LB_EINVAL, "fn must be 0..3 (got %s%lld)", "", (long long)fn);
  lb_status s = validate(dtype, v, v_stride, x, out, n, (int)mode);
  if (s != LB_OK || n == 0) return s;
  // default pieces of up to 2M pairs: log K on 8M pairs takes 1.00 ms end to
  // end against 0.98 (2^20), 1.20 (2^22) and 1.11 ms (2^24), one order and 20M
  // pairs 1.36 against 1.41, 1.48 and 1.65, per-pair orders and 220M pairs
  // 19.8 against 20.9, 19.5 and 20.2: larger ones leave longer first and last
  // copies unoverlapped, smaller ones cost more kernel ends
  // (FP32 the same bytes, 2^22 pairs: log I, 4M pairs, 246 us against 284 with
  // 2^21 and 269 with 2^24, 20M 993 / 1025 / 1008)
  if (chunk <= 0) chunk = (int64_t)1 << (dtype == LB_F64 ? 21 : 22);
  if (chunk > kChunk) chunk = kChunk;
  if ((fn >= 2 && dtype != LB_F64) || (fn == 3 && mode != LB_TIGHT))
    return fail(LB_ENOTSUP, "%sthe derivatives are implemented for LB_F64 (and LB_TIGHT for K) only", "", 0);
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return check_launch("cudaGetDevice");
  if (dev < 0 || dev >= kMaxDevices) return fail(LB_EINVAL, "device %s%lld out of range", "", (long long)dev);
  HostPipe& P = host_pipe(dev);
  std::lock_guard<std::mutex> lk(P.mu);
  if (!P.init && !host_pipe_init(P))
    return fail(LB_ENOMEM, "%slogbessel_host: stream or event creation failed", "", 0);
  const size_t es = dtype == LB_F64 ? 8 : 4;
  const int64_t nbuf = kHostSlots;                // copy-in, compute and copy-out of successive chunks overlap
  const int64_t cap = n < chunk ? n : chunk;
  const size_t vbytes = (size_t)(v_stride ? cap : 1) * es, xbytes = (size_t)cap * es;
  const size_t slot = ((vbytes + 255) & ~(size_t)255) + 2 * ((xbytes + 255) & ~(size_t)255);
  const size_t qbytes = (256 + 4 * (size_t)cap + 255) & ~(size_t)255;
  const size_t need = slot * nbuf + 2 * qbytes;   // + a K fallback queue per compute stream
  if (P.bytes < need) {
    if (P.dbuf) cudaFree(P.dbuf);
    P.dbuf = nullptr;
    P.bytes = 0;
    if (cudaMalloc((void**)&P.dbuf, need) != cudaSuccess) {
      cudaGetLastError();
      P.dbuf = nullptr;
      return fail(LB_ENOMEM, "%slogbessel_host: cudaMalloc of %lld bytes failed", "", (long long)need);
    }
    P.bytes = need;
  }
  cudaStream_t* st = P.st;
  // Pieces: chunk/8, chunk/4, chunk/2, then whole chunks, and from two chunks
  // on halves of what remains down to chunk/8, so that the first copy-in and
  // the last copy-out, which nothing overlaps, are short (halves from one chunk
  // on left a whole chunk and a scrap at some sizes: log I, 4M pairs, 604 us
  // against 493, d/dx 611 / 509); piece edges stay
  // on tile boundaries (chunk a multiple of 8 tiles), so the results equal
  // those of one pass.
  const bool ramp = chunk % (8 * kTile) == 0;
  int64_t cn = 0;
  for (int64_t c0 = 0, i = 0; s == LB_OK && c0 < n; c0 += cn, ++i) {
    const int64_t r = n - c0;
    cn = chunk;
    if (ramp) {
      if (i < 3) cn = chunk >> (3 - i);
      if (r <= chunk || (i >= 3 && r <= 2 * chunk)) {
        const int64_t half = (r / 2) / kTile * kTile;
        cn = half > chunk / 8 ? half : chunk / 8;
      }
    }
    if (cn > r) cn = r;
    const int b = (int)(i % nbuf);
    char* dv = P.dbuf + b * slot;
    char* dx = dv + ((vbytes + 255) & ~(size_t)255);
    char* dout = dx + ((xbytes + 255) & ~(size_t)255);
    const char* hv = (const char*)v + (v_stride ? c0 * (int64_t)es : 0);
    if ((i >= nbuf && cudaStreamWaitEvent(st[0], P.ev_out[b], 0) != cudaSuccess) ||   // slot b's results are out
        cudaMemcpyAsync(dv, hv, (size_t)(v_stride ? cn : 1) * es, cudaMemcpyHostToDevice, st[0]) != cudaSuccess ||
        cudaMemcpyAsync(dx, (const char*)x + c0 * (int64_t)es, (size_t)cn * es, cudaMemcpyHostToDevice, st[0]) != cudaSuccess ||
        cudaEventRecord(P.ev_in[b], st[0]) != cudaSuccess) {
      s = check_launch("logbessel_host: copy-in");
      break;
    }
    // one pass per chunk (cn <= cap <= kChunk), the K queue in ws.  Even and
    // odd pieces run on two compute streams with a queue each, so a piece's
    // kernels start while the previous piece's last kernels drain (the
    // blocks of the tile and K-integral kernels end at different times).
    cudaStream_t sc = st[(i & 1) ? 3 : 1];
    void* ws = P.dbuf + slot * nbuf + (size_t)(i & 1) * qbytes;
    if (cudaStreamWaitEvent(sc, P.ev_in[b], 0) != cudaSuccess) {
      s = check_launch("logbessel_host: copy-in");
      break;
    }
    if (dtype == LB_F32) {
      const float *fv = (const float*)dv, *fx = (const float*)dx;
      float* fo = (float*)dout;
      s = fn == 0 ? run_impl<KIND_I, false, float>(fv, v_stride, fx, fo, cn, (int)mode, -1, sc, nullptr, kChunk, n)
                  : run_impl<KIND_K, false, float>(fv, v_stride, fx, fo, cn, (int)mode, -1, sc, ws, kChunk, n);
    } else {
      const double *dvv = (const double*)dv, *dxx = (const double*)dx;
      double* dd = (double*)dout;
      switch (fn) {
        case 0: s = run_impl<KIND_I, false, double>(dvv, v_stride, dxx, dd, cn, (int)mode, -1, sc, nullptr, kChunk, n); break;
        case 1: s = run_impl<KIND_K, false, double>(dvv, v_stride, dxx, dd, cn, (int)mode, -1, sc, ws, kChunk, n); break;
        case 2: s = run_impl<KIND_I, true, double>(dvv, v_stride, dxx, dd, cn, (int)mode, -1, sc, nullptr, kChunk, n); break;
        default: s = run_impl<KIND_K, true, double>(dvv, v_stride, dxx, dd, cn, (int)mode, -1, sc, ws, kChunk, n); break;
      }
    }
    if (s != LB_OK) break;
    if (cudaEventRecord(P.ev_comp[b], sc) != cudaSuccess || cudaStreamWaitEvent(st[2], P.ev_comp[b], 0) != cudaSuccess ||
        cudaMemcpyAsync((char*)out + c0 * (int64_t)es, dout, (size_t)cn * es, cudaMemcpyDeviceToHost, st[2]) != cudaSuccess ||
        cudaEventRecord(P.ev_out[b], st[2]) != cudaSuccess) {
      s = check_launch("logbessel_host: copy-out");
      break;
    }
  }
  for (int i = 0; i < 4; ++i)
    if (cudaStreamSynchronize(st[i]) != cudaSuccess && s == LB_OK) s = check_launch("logbessel_host");
  // an asynchronous error of the last copies surfaces here, not in a later call
  if (s == LB_OK) s = check_launch("logbessel_host");
  return s;
}

lb_status logbessel_host_release(void) {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return check_launch("cudaGetDevice");
  if (dev < 0 || dev >= kMaxDevices) return fail(LB_EINVAL, "device %s%lld out of range", "", (long long)dev);
  HostPipe& P = host_pipe(dev);
  std::lock_guard<std::mutex> lk(P.mu);
  if (P.init) {
    for (int i = 0; i < 4; ++i) cudaStreamSynchronize(P.st[i]);
    host_pipe_destroy(P);
  }
  return LB_OK;
}

lb_status logbessel_check_status(unsigned int* bits, int clear) {
  if (!bits) return fail(LB_EINVAL, "%sNULL bits", "", 0);
  *bits = 0;
#ifdef LB_CHECKS
  unsigned int v = 0;
  if (cudaMemcpyFromSymbol(&v, lb_check_status, sizeof v) != cudaSuccess) return check_launch("logbessel_check_status");
  if (clear) {
    const unsigned int z = 0;
    if (cudaMemcpyToSymbol(lb_check_status, &z, sizeof z) != cudaSuccess) return check_launch("logbessel_check_status");
  }
  *bits = v;
  return LB_OK;
#else
  (void)clear;
  return fail(LB_ENOTSUP, "%sthis build has no index checks (build with LB_CHECKS)", "", 0);
#endif
}

const char* logbessel_last_error(void) { return g_last_error.c_str(); }

void logbessel_profile_enable(int on) {
  ProfState& P = prof();
  std::lock_guard<std::mutex> lk(P.mu);
  prof_drain_locked(P);
  if (on) {
    for (int i = 0; i < PS_NSLOTS; ++i) { P.ms[i] = 0.0; P.timed[i] = 0; }
  }
  P.on = on != 0;
}

int logbessel_profile_slots(void) { return PS_NSLOTS; }

lb_status logbessel_profile_get(int slot, const char** name, long long* launches, long long* timed_launches,
                                double* total_ms) {
  if (slot < 0 || slot >= PS_NSLOTS) return fail(LB_EINVAL, "profile slot %s%lld out of range", "", (long long)slot);
  ProfState& P = prof();
  std::lock_guard<std::mutex> lk(P.mu);
  prof_drain_locked(P);
  if (name) *name = kSlotNames[slot];
  if (launches) *launches = P.launches[slot];
  if (timed_launches) *timed_launches = P.timed[slot];
  if (total_ms) *total_ms = P.ms[slot];
  return LB_OK;
}

long long logbessel_launch_count(void) { return g_total_launches.load(); }

const char* logbessel_version(void) { return LB_VERSION; }

}  // extern "C"
