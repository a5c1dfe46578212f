// k_resample.cu -- resampling and redistribute on sm_103a.
//
//  * Quantisation of the weights to 64-bit fixed point, W_i = E(log w_i - m)
//    >> (62 - F), with exact 128-bit sums S, sum W^2, sum E (reduce pass; the
//    partial sums of eq. (7) from the rows, or from the move kernel's tile
//    records), the N_eff decision S^2 < N* sum W^2 (eq. (1) against the
//    threshold N* of Algorithm 2; 2 S^2 < N sum W^2 for N* = N/2), LSE_t and
//    log c_t (eqs. (2), (8)) in a single-block finaliser.
//  * Systematic resampling (MVR, Algorithm 4 line 1) on the integer CDF:
//    off_i = floor((N C_{i-1} + U)/S) is the exclusive cumulative sum of
//    ncopies and ncopies_i = off_{i+1} - off_i (eq. (9) holds by telescoping);
//    a block-local scan of W plus the block prefix gives C_i.
//  * Redistribute (Algorithm 5 as the definition of the output): output-tile
//    parallel gather.  The scan pass writes runstart[off_i] = i for every
//    survivor (a run of ncopies_i output rows starts at off_i) and the source
//    row of each tile's first output row; a tile of output rows loads its
//    slice of runstart (resetting it to -1 for the next iteration), a block
//    max-scan turns it into src(k), and the rows are copied with 16-byte
//    vector loads/stores.  Every tile does the same bounded work whatever the
//    weights.  Replaces the paper's MPI nearly-sort and rotational shifts
//    (Sec. 4) with O(1) passes over the data.
#include <atomic>
#include <cmath>

#include "particle_bodies.cuh"
#include "smc_internal.cuh"
#include "smc_kernels.h"

namespace smc {

// Tables of the fixed-point exponential: [0, 64) ~2^63 2^(-j/64),
// [64, 128) ~2^63 2^(-j/4096).
__constant__ uint64_t c_T[128];

// floor(sqrt(n)) for n < 2^126 by Newton's iteration from above.
static uint64_t isqrt_newton(u128 n) {
  if (n == 0) return 0;
  u128 x = u128(1) << 64;  // >= sqrt(n) for n < 2^128
  while (true) {
    const u128 y = (x + n / x) >> 1;
    if (y >= x) break;
    x = y;
  }
  return uint64_t(x);
}

// c_0 = 2^62, c_b = isqrt(c_{b-1} 2^63) ~= 2^63 2^(-2^-b) for b = 1..12;
// T1[j] (T[j]) is the product of c_1..c_6 over the set bits of j (c_1 for the
// top bit), T2[j] (T[64 + j]) the same with c_7..c_12; every product is
// floored to 2^63 fixed point.
static void build_table(uint64_t T[128]) {
  uint64_t c[13];
  c[0] = 1ull << 62;
  for (int b = 1; b <= 12; ++b) c[b] = isqrt_newton(u128(c[b - 1]) << 63);
  for (int half = 0; half < 2; ++half) {
    for (int j = 0; j < 64; ++j) {
      uint64_t acc = 1ull << 63;
      for (int b = 1; b <= 6; ++b)
        if (j & (1 << (6 - b))) acc = uint64_t((u128(acc) * c[6 * half + b]) >> 63);
      T[64 * half + j] = acc;
    }
  }
}

cudaError_t upload_expfx_table() {
  static bool done[64] = {false};
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev >= 0 && dev < 64 && done[dev]) return cudaSuccess;
  uint64_t T[128];
  build_table(T);
  e = cudaMemcpyToSymbol(c_T, T, sizeof T);
  if (e == cudaSuccess && dev >= 0 && dev < 64) done[dev] = true;
  return e;
}

// The device copy of the table on the current device, for the kernels of
// other translation units.
cudaError_t expfx_table(const uint64_t** out) {
  static std::atomic<const uint64_t*> at[64];
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  const bool kept = dev >= 0 && dev < 64;
  *out = kept ? at[dev].load() : nullptr;
  if (*out) return cudaSuccess;
  void* p = nullptr;
  e = cudaGetSymbolAddress(&p, c_T);
  if (e != cudaSuccess) return e;
  *out = static_cast<const uint64_t*>(p);
  if (kept) at[dev].store(*out);
  return cudaSuccess;
}

__device__ __forceinline__ void load_table(uint64_t* T) {
  if (threadIdx.x < 128) T[threadIdx.x] = c_T[threadIdx.x];
  __syncthreads();
}


// ---------------------------------------------------------------- state init
// reset value of Algorithm 4 line 3, -log N, from the exact log so that both
// implementations agree bit for bit
__global__ void k_state_init(DevState* st, int64_t n, int64_t t, int F) {
  chain_begin();
  if (threadIdx.x != 0) return;
  const double reset_logw = -det_log(double(n));
  st->t = t;
  st->cur = 0;
  st->flag = 0;
  st->err = 0;
  st->F = F;
  st->L = 1;
  st->m = 0.0;
  st->lse = 0.0;
  st->lse_prev = 0.0;
  st->logc = 0.0;
  st->ess = 0.0;
  st->reset_logw = reset_logw;
  st->S = st->U = 0;
  st->sw2_lo = st->sw2_hi = st->se_lo = st->se_hi = 0;
  st->recip = 0;
  st->rc_max = -INFINITY;
  st->rc_den = 0.0;
  for (int c = 0; c < kMaxD; ++c) st->rc_num[c] = st->mean[c] = 0.0;
  st->est_s = 0.0;
  st->trace = nullptr;
  st->trace_t0 = 0;
  st->mean_out = st->fhat_out = st->cov_out = nullptr;
  st->want_cov = 0;
  st->w_uniform = 0;
  st->est_ready = 0;
  st->pending = 0;
  st->rs_dirty = 0;
  st->rs_w = 0;
  st->sub_ready = 0;
  st->mkey = kNoMaxKey;
  st->tickets = 0;
}

// ---------------------------------------------------------------- max of log w (stateless path)
// Raises st->mkey; NaN is an error.  Integer-ordered keys with every load of a
// thread in flight: FP64 comparisons and a count (two lanes per SM and clock
// each) took 155 us at N = 2^24, 27 now.
__global__ void __launch_bounds__(kQThreads) k_max_logw(const double* __restrict__ logw, int64_t n, DevState* st) {
  chain_begin();
  __shared__ long long shm[kQThreads / 32];
  MaxTracker mt;
  mt.init();
  const int64_t base = int64_t(blockIdx.x) * kQTile + threadIdx.x;
  double v[kQItems];
#pragma unroll
  for (int k = 0; k < kQItems; ++k) {
    const int64_t i = base + k * kQThreads;
    v[k] = i < n ? __ldg(logw + i) : -INFINITY;
  }
#pragma unroll
  for (int k = 0; k < kQItems; ++k) mt.add(v[k]);
  if (mt.nan) record_error(st, SMC_ENONFINITE);
  const long long wm = warp_max_ll(mt.best);
  if ((threadIdx.x & 31) == 0) shm[threadIdx.x >> 5] = wm;
  __syncthreads();
  if (threadIdx.x == 0) {
    long long m = shm[0];
    for (int w = 1; w < kQThreads / 32; ++w) m = shm[w] > m ? shm[w] : m;
    if (m > *const_cast<volatile long long*>(&st->mkey)) atomicMax(&st->mkey, m);
  }
}

// ---------------------------------------------------------------- quantise: reduce
// Per block of 4096 weights: the exact sums S = sum W, sum W^2, sum E, and
// (EST) the partial sums sum_i E_i x_i of the estimate of eq. (7), whose
// normalised weights are E_i / sum E (the fixed-point exp of log w_i - m).
__device__ __forceinline__ float u64_to_float_trunc(uint64_t v) {
  if (v == 0) return 0.0f;
  const int e = 63 - __clzll((long long)v);
  const uint32_t mant = e >= 23 ? uint32_t(v >> (e - 23)) : uint32_t(v << (23 - e));
  return __uint_as_float((uint32_t(e + 127) << 23) | (mant & 0x7FFFFFu));
}
__device__ __forceinline__ void weight_of(uint64_t E, float* w) { *w = u64_to_float_trunc(E); }
__device__ __forceinline__ void weight_of(uint64_t E, double* w) { *w = __ull2double_rn(E); }

// What a quantise pass starts from.  In smc_step's own iteration no kernel has
// run between the move and this pass: the maximum is still a key, a move that
// gathered a pending copy wrote the other buffer, and the eq. (7) records
// are there when the weights started uniform (k_iter_finalize then brings the
// state up to date).
__device__ __forceinline__ double pass_max(const QuantArgs& a) {
  return a.fused ? from_ordered_key(a.st->mkey) : a.st->m;
}
__device__ __forceinline__ bool pass_cur(const QuantArgs& a) {
  return a.fused ? (a.st->cur ^ a.st->pending) != 0 : a.st->cur != 0;
}
__device__ __forceinline__ bool pass_records(const QuantArgs& a) {
  return a.est_src && (a.fused ? a.st->w_uniform : a.st->est_ready);
}

// Loads of rows the kernel only reads (read-only path), or, in a kernel whose
// other blocks wrote them before a grid barrier, at the coherent level (L2).
template <bool COH, typename V>
__device__ __forceinline__ V ld_rows(const V* p) {
  if constexpr (COH)
    return __ldcg(p);
  else
    return __ldg(p);
}

template <bool COH, typename V>
__device__ __forceinline__ V ld_plain(const V* p) {
  if constexpr (COH)
    return __ldcg(p);
  else
    return *p;
}

// eq. (7) partials of one quantise block from the move kernel's tile records
// {M_r, sum e^{log w - M_r} x} (FP32 samplers; one warp): scaled to the units
// of E_i (2^62 e^{log w - m}) and added over the block's tiles by a fixed
// shuffle tree.
__device__ __forceinline__ void quant_records(const QuantArgs& a, const int64_t blk) {
  constexpr int kTiles = kQTile / kEstTile;
  static_assert(kTiles <= 32, "one lane per tile record");
  const int lane = threadIdx.x & 31, d = a.d;
  const int64_t ntile = (a.n + kEstTile - 1) / kEstTile;
  const int64_t jt = blk * kTiles + lane;
  const bool have = lane < kTiles && jt < ntile && !a.st->err;
  const double* rec = a.epart + jt * (1 + d);
  const double Mr = have ? rec[0] : -INFINITY;
  const float f = Mr == -INFINITY ? 0.0f : __expf(float(Mr - pass_max(a))) * 0x1p62f;
  for (int c = 0; c < d; ++c) {
    const float v = warp_sum(have ? f * float(rec[1 + c]) : 0.0f);
    if (lane == 0) static_cast<float*>(a.xpart)[blk * d + c] = v;
  }
}

// Shared memory of one quantise-reduce block (declared by the calling kernel).
struct QuantReduceSmem {
  uint64_t T[128];
  uint64_t sh[kQThreads / 32][5];
  double shx[kQThreads / 32][32];
};

template <typename ST, int DMAX, bool EST, bool COH = false>
__device__ __forceinline__ void quant_reduce_body(const QuantArgs& a, const int blk, QuantReduceSmem& sm) {
  uint64_t* const T = sm.T;
  uint64_t (*const sh)[5] = sm.sh;
  double (*const shx)[32] = sm.shx;
  load_table(T);
  const DevState* st = a.st;
  if (blk == 0 && threadIdx.x == 0) a.st->sub_ready = 0;  // (no prefixes inside the tiles from this pass)
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  // rows shared by lanes (see below): 16-byte groups of kV columns
  constexpr int kV = 16 / sizeof(ST), kLanes = DMAX / kV > 0 ? DMAX / kV : 1, kRowsPer = 32 / kLanes;
  // (not for FP32 rows of 16: with this route the kernel needs 80 registers
  // instead of 64, and the records route below, which these samplers take
  // whenever they resample, 0.149 instead of 0.129 ms at N = 2^24)
  constexpr bool kShared = EST && !COH && DMAX >= 2 * kV && !(sizeof(ST) == 4 && DMAX == 16);
  bool shared_rows = false;
  uint64_t sw = 0;
  u128 sw2 = 0, se = 0;
  ST acc[DMAX];
#pragma unroll
  for (int c = 0; c < DMAX; ++c) acc[c] = ST(0);
  const int d = a.d;
  // eq. (7) from the move kernel's tile records when it wrote them this
  // iteration, else from the rows
  const bool use_rec = EST && pass_records(a);
  if (!st->err) {
    const double m = pass_max(a);
    const int sh_w = 62 - st->F;
    const int64_t base = int64_t(blk) * kQTile;
    const ST* __restrict__ x = static_cast<const ST*>(pass_cur(a) ? a.x[1] : a.x[0]);
    bool done = false;
    if constexpr (sizeof(ST) == 4) {  // (records exist for FP32 samplers only)
      if (use_rec) {
        // only log w is read: every load of the thread first (more bytes in
        // flight), then the arithmetic
        double lv[kQItems];
#pragma unroll
        for (int k = 0; k < kQItems; ++k) {
          const int64_t i = base + k * kQThreads + threadIdx.x;
          lv[k] = i < a.n ? a.logw[i] : 0.0;
        }
#pragma unroll
        for (int k = 0; k < kQItems; ++k) {
          const int64_t i = base + k * kQThreads + threadIdx.x;
          if (i < a.n) {
            const uint64_t E = expfx_a(__dsub_rn(m, lv[k]), T);
            const uint64_t W = E >> sh_w;
            a.wbuf[i] = W;
            sw += W;
            sw2 += u128(W) * W;
            se += E;
          }
        }
        done = true;
      }
    }
    if constexpr (COH && EST && DMAX <= 8) {
      // (the fused small-sampler iteration, rows written by other blocks of
      // the same launch: coherent loads, latency-bound) each group of four
      // items' log w and rows loaded first, then the arithmetic in the
      // same order as below
      if (!done && !use_rec) {
        for (int k0 = 0; k0 < kQItems; k0 += 4) {
          double lv[4];
          ST xr[4][DMAX];
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            const int64_t i = base + (k0 + u) * kQThreads + threadIdx.x;
            lv[u] = i < a.n ? __ldcg(a.logw + i) : 0.0;
#pragma unroll
            for (int c = 0; c < DMAX; ++c) xr[u][c] = (i < a.n && c < d) ? __ldcg(x + i * d + c) : ST(0);
          }
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            const int64_t i = base + (k0 + u) * kQThreads + threadIdx.x;
            if (i < a.n) {
              const uint64_t E = expfx_a(__dsub_rn(m, lv[u]), T);
              const uint64_t W = E >> sh_w;
              a.wbuf[i] = W;
              sw += W;
              sw2 += u128(W) * W;
              se += E;
              ST w;
              weight_of(E, &w);
#pragma unroll
              for (int c = 0; c < DMAX; ++c)
                if (c < d) acc[c] = fma(w, xr[u][c], acc[c]);
            }
          }
        }
        done = true;
      }
    }
    if constexpr (kShared) {
      if (!done && !use_rec && d == DMAX) {
        // kLanes lanes share a row, 16 bytes each, so that a warp's load covers
        // whole 128-byte lines: the warp's 32 rows of one k come in kLanes
        // loads of 32 / kLanes rows, lane l holding columns kV (l % kLanes) ..
        // of rows kRowsPer j + l / kLanes, j = 0 .. kLanes - 1.  (A thread
        // reading its own row touches 32 lines per load, kLanes times over:
        // 54 instead of 31 us at N = 2^20, D = 32.)
        const int lr = lane / kLanes, lc = lane % kLanes;
        const int64_t i0 = base + (threadIdx.x - lane) + lr;  // row of (k, j): i0 + 256 k + kRows j
        const bool whole = base + kQTile <= a.n;
        constexpr int kUnroll = DMAX * sizeof(ST) > 128 ? 1 : 2;
#pragma unroll kUnroll
        for (int k = 0; k < kQItems; ++k) {
          const int64_t i = base + k * kQThreads + threadIdx.x;
          float4 f[kLanes];
#pragma unroll
          for (int j = 0; j < kLanes; ++j) {
            const int64_t r = i0 + k * kQThreads + j * kRowsPer;
            f[j] = (whole || r < a.n) ? ld_rows<COH>(reinterpret_cast<const float4*>(x + r * DMAX) + lc)
                                      : make_float4(0.f, 0.f, 0.f, 0.f);
          }
          ST w = ST(0);
          if (i < a.n) {
            const uint64_t E = expfx_a(__dsub_rn(m, ld_plain<COH>(a.logw + i)), T);
            const uint64_t W = E >> sh_w;
            a.wbuf[i] = W;
            sw += W;
            sw2 += u128(W) * W;
            se += E;
            weight_of(E, &w);
          }
#pragma unroll
          for (int j = 0; j < kLanes; ++j) {
            const ST wj = __shfl_sync(0xffffffffu, w, j * kRowsPer + lr);
            const bool in = whole || i0 + k * kQThreads + j * kRowsPer < a.n;
            if constexpr (sizeof(ST) == 4) {
              const float g[4] = {f[j].x, f[j].y, f[j].z, f[j].w};
#pragma unroll
              for (int u = 0; u < kV; ++u)
                if (in) acc[j * kV + u] = fma(wj, ST(g[u]), acc[j * kV + u]);
            } else {
              const double g[2] = {__hiloint2double(__float_as_int(f[j].y), __float_as_int(f[j].x)),
                                   __hiloint2double(__float_as_int(f[j].w), __float_as_int(f[j].z))};
#pragma unroll
              for (int u = 0; u < kV; ++u)
                if (in) acc[j * kV + u] = fma(wj, ST(g[u]), acc[j * kV + u]);
            }
          }
        }
        done = true;
        shared_rows = true;
      }
    }
    if (!done)
#pragma unroll 4
    for (int k = 0; k < kQItems; ++k) {
      const int64_t i = base + k * kQThreads + threadIdx.x;
      if (i < a.n) {
        const uint64_t E = expfx_a(__dsub_rn(m, ld_plain<COH>(a.logw + i)), T);
        const uint64_t W = E >> sh_w;
        a.wbuf[i] = W;
        sw += W;
        sw2 += u128(W) * W;
        se += E;
        if (EST && !use_rec) {
          ST w;
          weight_of(E, &w);
          const ST* row = x + i * d;
          if (d == DMAX && (DMAX * sizeof(ST)) % 16 == 0) {
#pragma unroll
            for (int v = 0; v < int(DMAX * sizeof(ST) / 16); ++v) {
              const float4 f = ld_rows<COH>(reinterpret_cast<const float4*>(row) + v);
              const ST* fv = reinterpret_cast<const ST*>(&f);
#pragma unroll
              for (int u = 0; u < int(16 / sizeof(ST)); ++u) {
                const int c = v * int(16 / sizeof(ST)) + u;
                acc[c] = fma(w, fv[u], acc[c]);
              }
            }
          } else {
#pragma unroll
            for (int c = 0; c < DMAX; ++c)
              if (c < d) acc[c] = fma(w, ld_plain<COH>(row + c), acc[c]);
          }
        }
      }
    }
  }
  sw = warp_sum(sw);
  sw2 = warp_sum_u128(sw2);
  se = warp_sum_u128(se);
  if (lane == 0) {
    sh[wid][0] = sw;
    sh[wid][1] = uint64_t(sw2);
    sh[wid][2] = uint64_t(sw2 >> 64);
    sh[wid][3] = uint64_t(se);
    sh[wid][4] = uint64_t(se >> 64);
  }
  if (EST && !use_rec) {
    // warp sums in the state precision (the FP64 pipe is scarce), then FP64
    if (kShared && shared_rows) {
      // the shuffle tree of warp_sum over the 32 rows (offsets 16, 8, 4, 2, 1):
      // the high bits of a row's place are the lane's own j
      if constexpr (kShared) {
#pragma unroll
        for (int h = kLanes / 2; h > 0; h >>= 1)
#pragma unroll
          for (int j = 0; j < kLanes; ++j)
            if (j < h) {
#pragma unroll
              for (int u = 0; u < kV; ++u) acc[j * kV + u] += acc[(j + h) * kV + u];
            }
#pragma unroll
        for (int u = 0; u < kV; ++u) {
          ST v = acc[u];
#pragma unroll
          for (int o = 16; o >= kLanes; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
          if (lane < kLanes) shx[wid][lane * kV + u] = double(v);
        }
      }
    } else {
#pragma unroll
      for (int c = 0; c < DMAX; ++c) {
        if (c < d) {
          const ST v = warp_sum(acc[c]);
          if (lane == 0) shx[wid][c] = double(v);
        }
      }
    }
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    uint64_t tw = 0;
    u128 t2 = 0, te = 0;
    for (int w = 0; w < kQThreads / 32; ++w) {
      tw += sh[w][0];
      t2 += (u128(sh[w][2]) << 64) | sh[w][1];
      te += (u128(sh[w][4]) << 64) | sh[w][3];
    }
    uint64_t* q = a.qpart + 5 * int64_t(blk);
    q[0] = tw;
    q[1] = uint64_t(t2);
    q[2] = uint64_t(t2 >> 64);
    q[3] = uint64_t(te);
    q[4] = uint64_t(te >> 64);
  }
  if (EST && !use_rec && threadIdx.x < d) {
    double v = 0.0;
    for (int w = 0; w < kQThreads / 32; ++w) v += shx[w][threadIdx.x];
    static_cast<ST*>(a.xpart)[int64_t(blk) * d + threadIdx.x] = ST(v);
  }
  if (use_rec && wid == 0) quant_records(a, blk);
}

template <typename ST, int DMAX, bool EST>
__global__ void __launch_bounds__(kQThreads) k_quant_reduce(QuantArgs a) {
  chain_begin();
  __shared__ QuantReduceSmem sm;
  quant_reduce_body<ST, DMAX, EST>(a, blockIdx.x, sm);
}

// ---------------------------------------------------------------- quantise: reduce over clusters
// The same pass for samplers of few tiles.  With one block per tile of 4096
// weights a sampler of N = 20000 (D = 32) keeps 5 SMs busy with 16 rows per
// thread one after another (41 us, all of it latency).  Here a cluster of
// eight blocks shares a tile: block s quantises items [512 s, 512 s + 512)
// and forms the eq. (7) sums of the threads 32 s .. 32 s + 31 of the one-block
// pass (their rows: 256 k + 32 s + lane), one group of columns per warp with
// every row load in flight; block 0 combines the eight through distributed
// shared memory.  Every floating-point sum keeps the one-block pass's order
// (k ascending per thread, the shuffle tree, then the warps in order), so the
// results are the same bits.  csub receives the exclusive prefix of the
// 512-item sums inside the tile, for a scan of 512 items per block.
struct QuantClusterSmem {
  uint64_t T[128];
  uint64_t sh[kQThreads / 32][5];
  uint64_t part[kQSplit][5];       // rank 0: the blocks' integer sums
  double shx[kQSplit][kMaxD];      // rank 0: the blocks' column sums
  double w[kQTile / kQSplit];      // this block's eq. (7) weights, in the state's type
};

__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// The same barrier in two halves, for the start: shared memory of another
// block may only be accessed once that block runs.  Arriving on entry and
// waiting just before the first such access leaves the work between them to
// hide the wait.
__device__ __forceinline__ void cluster_arrive_started() {
  asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_wait_started() {
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// Stores v at p's place in the shared memory of the cluster's block 0, which
// has started (cluster_wait_started).
__device__ __forceinline__ void st_rank0(uint64_t* p, uint64_t v) {
  uint32_t a;
  asm volatile("mapa.shared::cluster.u32 %0, %1, 0;" : "=r"(a) : "r"(uint32_t(__cvta_generic_to_shared(p))));
  asm volatile("st.shared::cluster.u64 [%0], %1;" ::"r"(a), "l"(v) : "memory");
}

// The CW columns from c on of one row (as vectors when vec: d is a multiple
// of CW, so that every such group is aligned and complete).
template <int CW>
__device__ __forceinline__ void load_cols(const float* __restrict__ row, int c, int d, bool vec, float (&v)[CW]) {
  if (CW == 4 && vec) {
    const float4 f = __ldg(reinterpret_cast<const float4*>(row + c));
    v[0] = f.x;
    v[1 % CW] = f.y;
    v[2 % CW] = f.z;
    v[3 % CW] = f.w;
  } else if (CW == 2 && vec) {
    const float2 f = __ldg(reinterpret_cast<const float2*>(row + c));
    v[0] = f.x;
    v[1 % CW] = f.y;
  } else {
#pragma unroll
    for (int u = 0; u < CW; ++u) v[u] = c + u < d ? __ldg(row + c + u) : 0.0f;
  }
}
template <int CW>
__device__ __forceinline__ void load_cols(const double* __restrict__ row, int c, int d, bool vec, double (&v)[CW]) {
  if (CW >= 2 && vec) {
#pragma unroll
    for (int u = 0; u + 1 < CW; u += 2) {
      const double2 f = __ldg(reinterpret_cast<const double2*>(row + c + u));
      v[u] = f.x;
      v[u + 1] = f.y;
    }
  } else {
#pragma unroll
    for (int u = 0; u < CW; ++u) v[u] = c + u < d ? __ldg(row + c + u) : 0.0;
  }
}

template <typename ST, int CW, bool EST>
__global__ void __launch_bounds__(kQThreads, 2) __cluster_dims__(kQSplit, 1, 1) k_quant_reduce_cluster(QuantArgs a) {
  cluster_arrive_started();
  chain_begin();
  __shared__ QuantClusterSmem sm;
  const int s = int(cluster_rank());
  const int64_t tile = blockIdx.x / kQSplit;
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  DevState* st = a.st;
  const int d = a.d;
  const int64_t n = a.n, base = tile * kQTile;
  const bool use_rec = EST && pass_records(a);
  const bool rows = EST && !use_rec;
  const bool live = !st->err;
  // the rows first: their loads do not wait for the weights
  constexpr int kK = kQItems;                                     // rows per lane
  constexpr int kG = CW * sizeof(ST) > 16 ? kK / 2 : kK;          // of them in flight
  const int c0 = wid * CW;
  const bool mine = rows && live && c0 < d;
  const bool vec = d % CW == 0;
  const ST* __restrict__ x = static_cast<const ST*>(pass_cur(a) ? a.x[1] : a.x[0]);
  const int64_t r0 = base + 32 * s + lane;  // row of k: r0 + 256 k
  ST xr[EST ? kG : 1][CW];
  if constexpr (EST) {
    if (mine) {
#pragma unroll
      for (int k = 0; k < kG; ++k) {
        const int64_t i = r0 + int64_t(k) * kQThreads;
        if (i < n) {
          load_cols<CW>(x + i * d, c0, d, vec, xr[k]);
        } else {
#pragma unroll
          for (int u = 0; u < CW; ++u) xr[k][u] = ST(0);
        }
      }
    }
  }
  load_table(sm.T);
  uint64_t sw = 0;
  u128 sw2 = 0, se = 0;
  ST* const w = reinterpret_cast<ST*>(sm.w);
  if (live) {
    const double m = pass_max(a);
    const int sh_w = 62 - st->F;
#pragma unroll
    for (int q = 0; q < kQTile / kQSplit / kQThreads; ++q) {
      const int64_t i = base + s * (kQTile / kQSplit) + q * kQThreads + tid;
      if (i < n) {
        const uint64_t E = expfx_a(__dsub_rn(m, a.logw[i]), sm.T);
        const uint64_t W = E >> sh_w;
        a.wbuf[i] = W;
        sw += W;
        sw2 += u128(W) * W;
        se += E;
      }
    }
    if (rows) {
#pragma unroll
      for (int q = 0; q < kQTile / kQSplit / kQThreads; ++q) {
        const int e = q * kQThreads + tid;  // weight of (k = e / 32, lane e % 32)
        const int64_t i = base + int64_t(e >> 5) * kQThreads + 32 * s + (e & 31);
        ST v = ST(0);
        if (i < n) weight_of(expfx_a(__dsub_rn(m, a.logw[i]), sm.T), &v);
        w[e] = v;
      }
    }
  }
  sw = warp_sum(sw);
  sw2 = warp_sum_u128(sw2);
  se = warp_sum_u128(se);
  if (lane == 0) {
    sm.sh[wid][0] = sw;
    sm.sh[wid][1] = uint64_t(sw2);
    sm.sh[wid][2] = uint64_t(sw2 >> 64);
    sm.sh[wid][3] = uint64_t(se);
    sm.sh[wid][4] = uint64_t(se >> 64);
  }
  __syncthreads();
  cluster_wait_started();  // every block of the cluster runs: block 0 may be written
  if (tid == 0) {
    uint64_t tw = 0;
    u128 t2 = 0, te = 0;
    for (int v = 0; v < kQThreads / 32; ++v) {
      tw += sm.sh[v][0];
      t2 += (u128(sm.sh[v][2]) << 64) | sm.sh[v][1];
      te += (u128(sm.sh[v][4]) << 64) | sm.sh[v][3];
    }
    st_rank0(&sm.part[s][0], tw);
    st_rank0(&sm.part[s][1], uint64_t(t2));
    st_rank0(&sm.part[s][2], uint64_t(t2 >> 64));
    st_rank0(&sm.part[s][3], uint64_t(te));
    st_rank0(&sm.part[s][4], uint64_t(te >> 64));
  }
  if constexpr (EST) {
    if (rows && c0 < d) {
      ST acc[CW];
#pragma unroll
      for (int u = 0; u < CW; ++u) acc[u] = ST(0);
      if (live) {
#pragma unroll
        for (int k = 0; k < kK; ++k) {
          if (k >= kG) {  // (wide FP64 rows: the second half, loaded as the first is used)
            const int64_t i = r0 + int64_t(k) * kQThreads;
            if (i < n) load_cols<CW>(x + i * d, c0, d, vec, xr[k - kG]);
          }
          if (r0 + int64_t(k) * kQThreads < n) {
#pragma unroll
            for (int u = 0; u < CW; ++u) acc[u] = fma(w[32 * k + lane], xr[k % kG][u], acc[u]);
          }
        }
      }
#pragma unroll
      for (int u = 0; u < CW; ++u) {
        const ST v = warp_sum(acc[u]);
        if (lane == 0 && c0 + u < d) st_rank0(reinterpret_cast<uint64_t*>(&sm.shx[s][c0 + u]), uint64_t(__double_as_longlong(double(v))));
      }
    }
  }
  cluster_sync();
  if (s) return;
  if (tid == 0) {
    uint64_t tw = 0;
    u128 t2 = 0, te = 0;
    for (int v = 0; v < kQSplit; ++v) {
      a.csub[tile * kQSplit + v] = tw;
      tw += sm.part[v][0];
      t2 += (u128(sm.part[v][2]) << 64) | sm.part[v][1];
      te += (u128(sm.part[v][4]) << 64) | sm.part[v][3];
    }
    uint64_t* q = a.qpart + 5 * tile;
    q[0] = tw;
    q[1] = uint64_t(t2);
    q[2] = uint64_t(t2 >> 64);
    q[3] = uint64_t(te);
    q[4] = uint64_t(te >> 64);
    if (tile == 0) st->sub_ready = 1;
  }
  if constexpr (EST) {
    if (rows && tid >= 32 && tid < 32 + d) {
      double v = 0.0;
      for (int k = 0; k < kQSplit; ++k) v += sm.shx[k][tid - 32];
      static_cast<ST*>(a.xpart)[tile * d + tid - 32] = ST(v);
    }
    if (use_rec && wid == 0) quant_records(a, tile);
  }
}

__device__ __forceinline__ double u128_to_double(u128 v) {
  return double(uint64_t(v >> 64)) * 0x1p64 + double(uint64_t(v));
}

// eq. (7)'s numerators sum_i E_i x_i from the per-block partial sums, into
// sxsum[kMaxD] (shared memory); the whole block takes part.
__device__ __forceinline__ void estimate_sums(const QuantArgs& a, double* tpart, double* sxsum) {
  const int nb = a.nblocks;
  // logical thread j (of kFinThreads, whatever the block size) sums column
  // j % d over rows j / d, j / d + stride / d, ... in a fixed order
  // (deterministic, and the same in one-sampler and batched launches), in
  // the particle precision (the FP64 pipe is scarce); the per-thread
  // partials are then added in order per column
  const int stride = (kFinThreads / a.d) * a.d;
  const int64_t total_words = int64_t(nb) * a.d;
  for (int lt = threadIdx.x; lt < kFinThreads; lt += blockDim.x) {
    double part = 0.0;
    if (lt < stride) {
      if (a.dtype == SMC_F64) {
        const double* xp = static_cast<const double*>(a.xpart);
        for (int64_t j = lt; j < total_words; j += stride) part += xp[j];
      } else {
        const float* xp = static_cast<const float*>(a.xpart);
        float v[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
        int64_t j = lt;
        const int64_t s1 = int64_t(stride), s8 = 8 * s1;
        // four rounds' loads in flight at once, then their additions in
        // round order (the same sums as one round at a time)
        for (; j + 3 * s8 + 7 * s1 < total_words; j += 4 * s8) {
          float tv[32];
#pragma unroll
          for (int r = 0; r < 32; ++r) tv[r] = xp[j + r * s1];
#pragma unroll
          for (int q = 0; q < 4; ++q)
#pragma unroll
            for (int u = 0; u < 8; ++u) v[u] += tv[8 * q + u];
        }
        for (; j + 7 * s1 < total_words; j += s8) {
#pragma unroll
          for (int u = 0; u < 8; ++u) v[u] += xp[j + u * s1];
        }
        for (; j < total_words; j += stride) v[0] += xp[j];
        part = double(((v[0] + v[1]) + (v[2] + v[3])) + ((v[4] + v[5]) + (v[6] + v[7])));
      }
    }
    tpart[lt] = part;
  }
  __syncthreads();
  // column c's stride / d partials (tpart[c + d j]) summed by warps
  // c, c + nw, ...: lane l adds j = l, l + 32, ... in order, then a fixed
  // shuffle tree -- deterministic, and a short FP64 dependency chain
  {
    const int per_col = stride / a.d;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
    for (int c = wid; c < a.d; c += nwarps) {
      double t = 0.0;
      for (int j = lane; j < per_col; j += 32) t += tpart[c + a.d * j];
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
      if (lane == 0) sxsum[c] = t;
    }
  }
  __syncthreads();
}

// ---------------------------------------------------------------- quantise: finalise
// Single block: totals, exclusive prefix of the block sums (the CDF base of
// each scan block), decision, systematic offset U, division constants, LSE,
// N_eff, log c_t, and the statistics record.
__device__ __forceinline__ void quant_finalize_body(const QuantArgs& a, const int set_lse_prev) {
  __shared__ uint64_t scratch[33];
  __shared__ uint64_t shw[32], sh2l[32], sh2h[32], shel[32], sheh[32];
  DevState* st = a.st;
  const int nb = a.nblocks;
  uint64_t tw = 0;
  u128 t2 = 0, te = 0;
#pragma unroll 4
  for (int b = threadIdx.x; b < nb; b += blockDim.x) {
    const uint64_t* q = a.qpart + 5 * int64_t(b);
    tw += q[0];
    t2 += (u128(q[2]) << 64) | q[1];
    te += (u128(q[4]) << 64) | q[3];
  }
  tw = warp_sum(tw);
  t2 = warp_sum_u128(t2);
  te = warp_sum_u128(te);
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
  if (lane == 0) {
    shw[wid] = tw;
    sh2l[wid] = uint64_t(t2);
    sh2h[wid] = uint64_t(t2 >> 64);
    shel[wid] = uint64_t(te);
    sheh[wid] = uint64_t(te >> 64);
  }
  // exclusive scan of the block sums of W: contiguous chunk per thread
  const int chunk = (nb + blockDim.x - 1) / blockDim.x;
  const int b0 = threadIdx.x * chunk, b1 = min(nb, b0 + chunk);
  uint64_t local = 0;
#pragma unroll 4
  for (int b = b0; b < b1; ++b) local += a.qpart[5 * int64_t(b)];
  uint64_t total;
  uint64_t pre = block_excl_scan_u64(local, scratch, &total);  // contains __syncthreads
  for (int b = b0; b < b1; ++b) {
    a.cbase[b] = pre;
    pre += a.qpart[5 * int64_t(b)];
  }
  // eq. (7): f_t = sum_i E_i x_i / sum_i E_i from the per-block partial sums
  __shared__ double sxsum[kMaxD];
  const bool est = a.x[0] != nullptr && a.d > 0;
  if (est) {
    __shared__ double tpart[kFinThreads];
    estimate_sums(a, tpart, sxsum);
  }
  // eq. (7): the weighted mean, one column per thread
  {
    u128 se_all = 0;
    for (int w = 0; w < nw; ++w) se_all += (u128(sheh[w]) << 64) | shel[w];
    const double se_all_d = u128_to_double(se_all);
    if (est && !st->err && se_all_d > 0.0 && int(threadIdx.x) < a.d) {
      double* const mean_out = st->mean_out;  // (loaded before the store below)
      const double mc = sxsum[threadIdx.x] / se_all_d;
      st->mean[threadIdx.x] = mc;
      if (mean_out) mean_out[threadIdx.x] = mc;
    }
  }
  // the totals, then three independent chains, each a long one on this GPU, on
  // three warps (on three lanes of one warp they ran one after another, and
  // the quotient was the compiler's 128-bit division; 13.6 -> 12.4 us for a
  // batch of 60): the quotient for the copy counts, the logarithm of LSE, the
  // division of N_eff
  __shared__ uint64_t s_R;
  __shared__ double s_lse, s_sed, s_ess;
  const uint64_t n = uint64_t(a.n);
  uint64_t S = 0;
  u128 sw2 = 0;
  if (lane == 0 && wid < 3) {
    for (int w = 0; w < nw; ++w) {
      S += shw[w];
      sw2 += (u128(sh2h[w]) << 64) | sh2l[w];
    }
    if (wid == 0) {
      // S >= 2^F = 2^(63 - ceil(log2 N)), so floor(N 2^64 / S) <= 2^(2 ceil(log2 N) + 1) fits 64 bits
      s_R = S > n ? quotient_2p64(n, S) : 0;
    } else if (wid == 1) {
      u128 se1 = 0;
      for (int w = 0; w < nw; ++w) se1 += (u128(sheh[w]) << 64) | shel[w];
      s_sed = u128_to_double(se1);
      s_lse = st->m + log(s_sed * 0x1p-62);
    } else {
      const double Sd = double(S);
      s_ess = (S && sw2) ? Sd * Sd / u128_to_double(sw2) : 0.0;
    }
  }
  __syncthreads();
  if (threadIdx.x) return;
  // the state the record needs, loaded before the first store (nothing else
  // writes these fields while this block finalises)
  const int err0 = st->err;
  const int64_t t_now = st->t, trace_t0 = st->trace_t0;
  const double m = st->m, lse_prev = st->lse_prev;
  smc_iter_stats* const trace = st->trace;
  u128 se = 0;
  for (int w = 0; w < nw; ++w) se += (u128(sheh[w]) << 64) | shel[w];
  const uint64_t R = s_R;
  const double lse = s_lse, se_d = s_sed, ess = s_ess;
  int flag = 0;
  if (!err0 && S > 0) {
    if (a.mode == SMC_RESAMPLE_ALWAYS)
      flag = 1;
    else if (a.mode == SMC_RESAMPLE_NEVER)
      flag = 0;
    else if (a.nstar > 0)  // N_eff < N*  <=>  S^2 < N* sum W^2 (Algorithm 2, line 7)
      flag = u128(S) * S < u128(uint64_t(a.nstar)) * sw2;
    else  // N* = N/2
      flag = (u128(S) * S * 2) < u128(n) * sw2;
  }
  const P4 r = stream_block(a.seed, uint64_t(t_now), kPurposeResample, 0xFFFFFFFFull, 0);
  const uint64_t r64 = (uint64_t(r.v[0]) << 32) | r.v[1];
  const uint64_t U = S ? __umul64hi(r64, S) : 0;
  const int L = S ? 64 - __clzll((long long)S) : 1;
  st->est_s = se_d * 0x1p-62;
  st->S = S;
  st->U = U;
  st->L = L;
  st->recip = R;
  st->sw2_lo = uint64_t(sw2);
  st->sw2_hi = uint64_t(sw2 >> 64);
  st->se_lo = uint64_t(se);
  st->se_hi = uint64_t(se >> 64);
  st->flag = flag;
  st->lse = lse;
  st->ess = ess;
  const double logc = lse - lse_prev;
  st->logc = logc;
  if (set_lse_prev) st->lse_prev = lse;
  smc_iter_stats rec;
  rec.lse = lse;
  rec.logc = logc;
  rec.ess = ess;
  rec.max_logw = m;
  rec.resampled = flag;
  rec.t = t_now;
  rec.survivors = 0;
  st->survivors = 0;
  st->last = rec;
  if (trace) {
    const int64_t idx = t_now - trace_t0 - 1;
    if (idx >= 0) trace[idx] = rec;
  }
  if (a.stats_out) *a.stats_out = rec;
}

__global__ void __launch_bounds__(kFinThreads) k_quant_finalize(QuantArgs a, int set_lse_prev) {
  quant_finalize_body(a, set_lse_prev);
}

// ---------------------------------------------------------------- an iteration of smc_step: finalise
// The single-block part that the scan waits for, and nothing else: the
// totals, the CDF base of every block, the decision, U and floor(N 2^64 / S),
// and the state's step from t - 1 to t.  What only the caller reads (LSE,
// N_eff, the mean, the recycling sums) is the scan launch's extra block
// (iter_stats), off the chain of kernels.  As begin + maximum + finalise + commit
// kernels, with the logarithm and divisions of the statistics in the chain,
// these steps took 22 us of an iteration whatever N.
__global__ void __launch_bounds__(kFinThreads) k_iter_finalize(QuantArgs a) {
  chain_begin();
  __shared__ uint64_t s_w[33], s_2l[32], s_2h[32], s_el[32], s_eh[32];
  DevState* st = a.st;
  const int nb = a.nblocks, tid = threadIdx.x, lane = tid & 31, wid = tid >> 5, nw = blockDim.x >> 5;
  // (each of the four threads at work in the end loads what it needs now)
  const bool role = lane == 0 && wid < 4;
  int wu = 0, pend = 0, cur = 0, rsw = 0, err = 0;
  int64_t t = 0, t0 = 0;
  long long key = 0;
  smc_iter_stats* trace = nullptr;
  if (role) {
    err = st->err;
    key = st->mkey;
    t = st->t + 1;
    if (wid == 3) {
      wu = st->w_uniform;
      pend = st->pending;
      cur = st->cur;
      rsw = st->rs_w;
      trace = st->trace;
      t0 = st->trace_t0;
    }
  }
  const int chunk = (nb + blockDim.x - 1) / blockDim.x;
  const int b0 = tid * chunk, b1 = min(nb, b0 + chunk);
  uint64_t tw = 0;
  u128 t2 = 0, te = 0;
#pragma unroll 4
  for (int b = b0; b < b1; ++b) {
    const uint64_t* q = a.qpart + 5 * int64_t(b);
    tw += q[0];
    t2 += (u128(q[2]) << 64) | q[1];
    te += (u128(q[4]) << 64) | q[3];
  }
  const uint64_t incl = warp_incl_scan_u64(tw);
  t2 = warp_sum_u128(t2);
  te = warp_sum_u128(te);
  if (lane == 31) s_w[wid] = incl;
  if (lane == 0) {
    s_2l[wid] = uint64_t(t2);
    s_2h[wid] = uint64_t(t2 >> 64);
    s_el[wid] = uint64_t(te);
    s_eh[wid] = uint64_t(te >> 64);
  }
  __syncthreads();
  uint64_t S = 0, pre = 0;  // every warp adds up the warps' totals it needs
  {
    const uint64_t v = lane < nw ? s_w[lane] : 0;
    const uint64_t vi = warp_incl_scan_u64(v);
    S = __shfl_sync(0xffffffffu, vi, 31);
    pre = __shfl_sync(0xffffffffu, vi - v, wid);
  }
  pre += incl - tw;
  for (int b = b0; b < b1; ++b) {
    a.cbase[b] = pre;
    pre += a.qpart[5 * int64_t(b)];
  }
  if (wid >= 4) return;
  u128 sw2 = 0, se = 0;
  if (wid == 1) sw2 = warp_sum_u128(lane < nw ? (u128(s_2h[lane]) << 64) | s_2l[lane] : u128(0));
  if (wid == 2) se = warp_sum_u128(lane < nw ? (u128(s_eh[lane]) << 64) | s_el[lane] : u128(0));
  if (!role) return;
  const double M = from_ordered_key(key);
  const bool bad = !(M > -INFINITY && M < INFINITY);
  const uint64_t n = uint64_t(a.n);
  if (wid == 0) {
    st->S = S;
    st->recip = S > n ? quotient_2p64(n, S) : 0;  // (S > N unless an error left no weight)
  } else if (wid == 1) {
    int flag = 0;
    if (!err && !bad && S > 0) {
      if (a.mode == SMC_RESAMPLE_ALWAYS)
        flag = 1;
      else if (a.mode == SMC_RESAMPLE_NEVER)
        flag = 0;
      else if (a.nstar > 0)  // N_eff < N*  <=>  S^2 < N* sum W^2 (Algorithm 2, line 7)
        flag = u128(S) * S < u128(uint64_t(a.nstar)) * sw2;
      else  // N* = N/2
        flag = (u128(S) * S * 2) < u128(n) * sw2;
    }
    st->flag = flag;
    st->sw2_lo = uint64_t(sw2);
    st->sw2_hi = uint64_t(sw2 >> 64);
  } else if (wid == 2) {
    const P4 r = stream_block(a.seed, uint64_t(t), kPurposeResample, 0xFFFFFFFFull, 0);
    const uint64_t r64 = (uint64_t(r.v[0]) << 32) | r.v[1];
    st->U = S ? __umul64hi(r64, S) : 0;
    st->L = S ? 64 - __clzll((long long)S) : 1;
    st->se_lo = uint64_t(se);
    st->se_hi = uint64_t(se >> 64);
  } else {
    if (bad) record_error(st, SMC_ENONFINITE);
    st->t = t;
    st->m = M;
    st->mkey = kNoMaxKey;
    // the move wrote eq. (7) records iff the weights it started from were
    // uniform; after its reweight they are not
    st->est_ready = wu;
    st->w_uniform = 0;
    // a move that gathered a deferred resampling's rows wrote them to the
    // other buffer, which is now current; the run starts it read stay set, so
    // the next scan writes the other array (which that move reset if it was
    // dirty) and this one is marked dirty
    if (pend) {
      st->cur = cur ^ 1;
      st->pending = 0;
      st->rs_w = rsw ^ 1;
      st->rs_dirty = 1;
    }
    st->survivors = 0;
    st->last.survivors = 0;
    if (trace && t - t0 - 1 >= 0) trace[t - t0 - 1].survivors = 0;
  }
}

// The iteration's statistics (one block, beside the scan's): LSE, N_eff, log
// c_t, the mean of eq. (7) and the recycling sums of eq. (6), each with the
// operations of quant_finalize_body and commit_warp in their order.
struct IterStatsSmem {
  double tpart[kFinThreads];
  double sxsum[kMaxD];
  double lse, ess;
};
__device__ __forceinline__ void iter_stats(const QuantArgs& a, IterStatsSmem& sm) {
  DevState* st = a.st;
  const int tid = threadIdx.x, last_warp = (blockDim.x >> 5) - 1;
  const double se_d = u128_to_double((u128(st->se_hi) << 64) | st->se_lo);
  // the two longest chains first, on warps of their own
  if (tid == 32 * last_warp) sm.lse = st->m + log(se_d * 0x1p-62);
  if (tid == 32 * (last_warp - 1)) {
    const double Sd = double(st->S);
    const u128 sw2 = (u128(st->sw2_hi) << 64) | st->sw2_lo;
    sm.ess = (st->S && sw2) ? Sd * Sd / u128_to_double(sw2) : 0.0;
  }
  const bool est = a.x[0] != nullptr && a.d > 0;
  if (est)
    estimate_sums(a, sm.tpart, sm.sxsum);
  else
    __syncthreads();
  if (tid >= 32) return;
  const int err = st->err, flag = st->flag;
  const int64_t t = st->t, t0 = st->trace_t0;
  const double m = st->m, lse_prev = st->lse_prev, rmax = st->rc_max, rden = st->rc_den;
  smc_iter_stats* const trace = st->trace;
  double* const fh = st->fhat_out;
  double* const mean_out = st->mean_out;
  const double lse = sm.lse, logc = lse - lse_prev;
  static_assert(kMaxD <= 32, "one column per lane");
  if (est && !err) {
    double mc = 0.0, rnum = 0.0;
    if (tid < a.d) {
      rnum = st->rc_num[tid];
      mc = se_d > 0.0 ? sm.sxsum[tid] / se_d : st->mean[tid];
    }
    const double M = fmax(rmax, logc);
    // (one of the two exponents is 0, and e^0 = 1)
    const double sc = (rmax == -INFINITY) ? 0.0 : (rmax == M ? 1.0 : exp(__dsub_rn(rmax, M)));
    const double e = logc == M ? 1.0 : exp(__dsub_rn(logc, M));
    const double den = __fma_rn(rden, sc, e);
    if (tid < a.d) {
      st->mean[tid] = mc;
      if (mean_out) mean_out[tid] = mc;
      const double num = __fma_rn(rnum, sc, __dmul_rn(e, mc));
      st->rc_num[tid] = num;
      if (fh) fh[tid] = __ddiv_rn(num, den);
    }
    __syncwarp();  // (every lane has read the sums' scale)
    if (tid == 0) {
      st->rc_den = den;
      st->rc_max = M;
    }
  }
  if (tid) return;
  st->est_s = se_d * 0x1p-62;
  st->lse = lse;
  st->ess = sm.ess;
  st->logc = logc;
  // LSE_t becomes the next LSE_{t-1}, 0 after a reset
  st->lse_prev = (flag && !err) ? 0.0 : lse;
  // (survivors: the finaliser zeroed it, the end of the iteration sets it)
  const int64_t idx = t - t0 - 1;
  smc_iter_stats* const recs[2] = {&st->last, trace && idx >= 0 ? trace + idx : nullptr};
#pragma unroll
  for (int k = 0; k < 2; ++k) {
    if (!recs[k]) continue;
    recs[k]->lse = lse;
    recs[k]->logc = logc;
    recs[k]->ess = sm.ess;
    recs[k]->max_logw = m;
    recs[k]->resampled = flag;
    recs[k]->t = t;
  }
  if (a.stats_out) {
    smc_iter_stats r;
    r.lse = lse;
    r.logc = logc;
    r.ess = sm.ess;
    r.max_logw = m;
    r.resampled = flag;
    r.t = t;
    r.survivors = 0;
    *a.stats_out = r;
  }
}

// The end of an iteration, by the last block of its last kernel to finish (so
// that every block has read the state it changes): a resampled iteration's
// copy becomes current, or pending when the next move makes it.  All threads
// of every block call it once.
__device__ __forceinline__ void end_iteration(DevState* st, unsigned blocks, int defer) {
  __syncthreads();
  if (threadIdx.x) return;
  __threadfence();
  if (atomicAdd(&st->tickets, 1u) != blocks - 1) return;
  __threadfence();
  st->tickets = 0;
  if (!st->flag || st->err) return;
  const int64_t surv = int64_t(*const_cast<volatile unsigned long long*>(&st->survivors));
  st->last.survivors = surv;
  const int64_t idx = st->t - st->trace_t0 - 1;
  if (st->trace && idx >= 0) st->trace[idx].survivors = surv;
  st->w_uniform = 1;  // a resampled iteration leaves every log w at reset_logw
  if (defer)
    st->pending = 1;
  else
    st->cur ^= 1;
}

// ---------------------------------------------------------------- copy-tile sources
// Every redistribute tile whose first output row k lies in a survivor's run
// [lo, hi) gets src = that survivor.  A thread writes the tile starts of its
// own short runs; a run spanning more than kBigRun tile starts (a heavily
// copied particle: in the one-hot case one run covers all N rows) is queued
// and written by the whole block after a barrier.  Every thread of the block
// must call tile_starts_flush.
constexpr int kBigRun = 4;
constexpr int kBigRuns = 64;
struct BigRuns {
  int count;
  int32_t src[kBigRuns];
  int64_t first[kBigRuns];  // first tile index
  int64_t tiles[kBigRuns];  // tile starts in the run
};

__device__ __forceinline__ void tile_starts_of_run(int32_t* __restrict__ tile_src, uint64_t lo, uint64_t hi,
                                                   uint64_t n, int32_t i, BigRuns& big) {
  const int sh = src_shift(int64_t(n));
  const uint64_t rows = 1ull << sh;
  const uint64_t kb0 = (lo + rows - 1) & ~(rows - 1);
  const uint64_t end = hi < n ? hi : n;
  if (kb0 >= end) return;
  const uint64_t tiles = (end - kb0 + rows - 1) >> sh;
  if (tiles > uint64_t(kBigRun)) {
    const int slot = atomicAdd(&big.count, 1);
    if (slot < kBigRuns) {
      big.src[slot] = i;
      big.first[slot] = int64_t(kb0 >> sh);
      big.tiles[slot] = int64_t(tiles);
      return;
    }
  }
  for (uint64_t kb = kb0; kb < end; kb += rows) tile_src[kb >> sh] = i;  // (short run, or the queue is full)
}

__device__ __forceinline__ void tile_starts_flush(int32_t* __restrict__ tile_src, BigRuns& big) {
  __syncthreads();
  const int nb = min(big.count, kBigRuns);
  for (int r = 0; r < nb; ++r)
    for (int64_t t = threadIdx.x; t < big.tiles[r]; t += blockDim.x) tile_src[big.first[r] + t] = big.src[r];
}

// ---------------------------------------------------------------- quantise: scan + ncopies
// Shared memory of the scan: the block's W staged for a blocked layout (then
// its copy counts), the block scan's scratch and the long-run queue.
struct ScanSmem {
  struct {
    uint64_t w[kQThreads * 17];
  } buf;
  uint64_t scratch[33];
  BigRuns big;
};

// ITEMS consecutive items per thread (a block covers kQThreads ITEMS items):
// kQItems for the quantise blocks of kQTile; fewer for a sampler whose N fits
// one block of kQThreads ITEMS items (shorter per-thread chains, the same
// exact integers).
// base: the block's first item; C0: the exclusive prefix of W before it.
template <int ITEMS = kQItems>
__device__ __forceinline__ void quant_scan_body(const QuantArgs& a, const int64_t base, const uint64_t C0, ScanSmem& sm) {
  static_assert(ITEMS >= 1 && ITEMS <= kQItems, "items per thread");
  const DevState* st = a.st;
  if (st->err || !(a.force || st->flag)) return;
  auto& buf = sm.buf;
  uint64_t* const scratch = sm.scratch;
  BigRuns& big = sm.big;
  if (threadIdx.x == 0) big.count = 0;
  const int64_t n = a.n;
  // the quantised weights of the reduce pass, staged for a blocked layout
#pragma unroll 4
  for (int k = 0; k < ITEMS; ++k) {
    const int idx = k * kQThreads + threadIdx.x;
    const int64_t i = base + idx;
    buf.w[(idx / ITEMS) * (ITEMS + 1) + idx % ITEMS] = i < n ? a.wbuf[i] : 0ull;
  }
  __syncthreads();
  const uint64_t S = st->S, U = st->U;
  uint64_t* const mine = buf.w + threadIdx.x * (ITEMS + 1);
  uint64_t tsum = 0;
#pragma unroll
  for (int q = 0; q < ITEMS; ++q) tsum += mine[q];
  uint64_t btot;
  const uint64_t C = C0 + block_excl_scan_u64(tsum, scratch, &btot);
  unsigned nsurv = 0;
  // off_i = floor((N C_{i-1} + U) / S): the estimate mulhi(C, floor(N 2^64/S))
  // is at most 2 below floor(N C / S), and floor((N C + U)/S) is at most 1
  // above that; exact 128-bit comparisons fix the result.
  const uint64_t Rn = st->recip;  // floor(N 2^64 / S)
  // the run-start array, chosen once (its choice does not change during the
  // pass; read per store, it was a load after every store)
  int32_t* const rsa = rs_now(a.runstart, a.runstart_alt, st);
  auto quot = [&](uint64_t c) -> uint64_t {
    const u128 X = u128(n) * c + U;
    uint64_t qq = __umul64hi(c, Rn);
    u128 nxt = u128(qq + 1) * S;
#pragma unroll
    for (int it = 0; it < 3; ++it)
      if (nxt <= X) {
        ++qq;
        nxt += S;
      }
    return qq;
  };
  // the items one after another, each offset computed as it is needed, from a
  // short loop (ITEMS + 1 unrolled quotients overflow the instruction cache:
  // 125 instead of 96 us at N = 2^24 with copy counts)
  const int64_t i0 = base + int64_t(threadIdx.x) * ITEMS;
  const bool counts = a.ncopies != nullptr;
  uint64_t cp = C, op = quot(C);
#pragma unroll 4
  for (int q = 0; q < ITEMS; ++q) {
    const uint64_t cn = cp + mine[q];
    const uint64_t on = quot(cn);
    const int64_t i = i0 + q;
    if (counts) mine[q] = on - op;  // (the item's own W is done with)
    if (on > op && i < n) {
      ++nsurv;
      if (a.write_rs) {  // (copy counts alone need no run starts or tile sources)
        rsa[op] = int32_t(i);
        tile_starts_of_run(a.tile_src, op, on, uint64_t(n), int32_t(i), big);
      }
    }
    cp = cn;
    op = on;
  }
  tile_starts_flush(a.tile_src, big);  // (block barrier inside)
  unsigned v = nsurv;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  if ((threadIdx.x & 31) == 0 && v) atomicAdd(&const_cast<DevState*>(st)->survivors, (unsigned long long)v);
  if (counts) {
#pragma unroll 4
    for (int k = 0; k < ITEMS; ++k) {
      const int idx = k * kQThreads + threadIdx.x;
      const int64_t i = base + idx;
      if (i < n) a.ncopies[i] = int32_t(buf.w[(idx / ITEMS) * (ITEMS + 1) + idx % ITEMS]);
    }
  }
}

__global__ void __launch_bounds__(kQThreads, 4) k_quant_scan(QuantArgs a) {
  __shared__ ScanSmem sm;
  quant_scan_body(a, int64_t(blockIdx.x) * kQTile, a.cbase[blockIdx.x], sm);
}

// 512 items per block (samplers of few tiles: eight times the blocks and two
// quotients per thread instead of sixteen).  The prefix inside the tile comes
// from the cluster reduce; when another reduce wrote W (a batch's), from W.
__global__ void __launch_bounds__(kQThreads, 4) k_quant_scan_sub(QuantArgs a) {
  constexpr int kSub = kQTile / kQSplit;
  __shared__ ScanSmem sm;
  const int64_t tile = blockIdx.x / kQSplit, base = int64_t(blockIdx.x) * kSub;
  if (base >= a.n || a.st->err || !(a.force || a.st->flag)) return;
  uint64_t C0 = a.cbase[tile];
  if (a.st->sub_ready) {
    C0 += a.csub[blockIdx.x];
  } else {
    uint64_t v = 0, total;
    for (int64_t i = tile * kQTile + threadIdx.x; i < base; i += kQThreads) v += a.wbuf[i];
    block_excl_scan_u64(v, sm.scratch, &total);
    C0 += total;
  }
  quant_scan_body<kSub / kQThreads>(a, base, C0, sm);
}

// The scan of an iteration of smc_step (SUB: 512 items per block), its
// statistics in the first block (so that they run beside the scan, not after
// it: as the last block they ended a scan of 4096 blocks 10 us later).
template <bool SUB>
__global__ void __launch_bounds__(kQThreads, 4) k_iter_scan(QuantArgs a) {
  chain_begin();
  __shared__ union {
    ScanSmem scan;
    IterStatsSmem stats;
  } sm;
  const int blk = int(blockIdx.x) - 1;
  if (blk < 0) {
    iter_stats(a, sm.stats);
  } else if constexpr (SUB) {
    constexpr int kSub = kQTile / kQSplit;
    const int64_t base = int64_t(blk) * kSub;
    if (base < a.n && !a.st->err && (a.force || a.st->flag))
      quant_scan_body<kSub / kQThreads>(a, base, a.cbase[blk / kQSplit] + a.csub[blk], sm.scan);
  } else {
    quant_scan_body(a, int64_t(blk) * kQTile, a.cbase[blk], sm.scan);
  }
  if (a.defer) end_iteration(a.st, gridDim.x, 1);
}

// ---------------------------------------------------------------- standalone ncopies scan
// Thread t of a block owns the 16 consecutive entries [base + 16 t, +16) of
// the caller's ncopies, read with 16-byte loads when the vector is 16-byte
// aligned and the group is complete (scalar loads otherwise).
__device__ __forceinline__ void load_counts(const int32_t* __restrict__ nc, int64_t n, int64_t first, int32_t c[16]) {
  const bool vec = ((reinterpret_cast<uintptr_t>(nc) & 15) == 0) && first + 16 <= n;
  if (vec) {
    const int4* p = reinterpret_cast<const int4*>(nc + first);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int4 v = __ldg(p + q);
      c[4 * q] = v.x;
      c[4 * q + 1] = v.y;
      c[4 * q + 2] = v.z;
      c[4 * q + 3] = v.w;
    }
  } else {
#pragma unroll
    for (int q = 0; q < 16; ++q) c[q] = first + q < n ? nc[first + q] : 0;
  }
}

// A block's sum of copy counts carries this bit when a count was negative.
constexpr uint64_t kNcBad = 1ull << 63;

// The outcome of the checks: SMC_EINVAL recorded, or (stateless calls, whose
// error word starts with the call) set to what was found.
__device__ __forceinline__ void nc_verdict(const NcScanArgs& a, bool bad) {
  if (a.reset_err)
    a.st->err = bad ? SMC_EINVAL : SMC_OK;
  else if (bad)
    record_error(a.st, SMC_EINVAL);
}

// Exclusive prefix of the block sums (cbase) and the check sum == n.
__device__ __forceinline__ void nc_finalize_body(const NcScanArgs& a) {
  __shared__ uint64_t scratch[33];
  const int nb = a.nblocks;
  const int chunk = (nb + blockDim.x - 1) / blockDim.x;
  const int b0 = threadIdx.x * chunk, b1 = min(nb, b0 + chunk);
  uint64_t local = 0;
  bool bad = false;
  for (int b = b0; b < b1; ++b) {
    const uint64_t v = a.part[b];
    local += v & ~kNcBad;
    bad |= (v & kNcBad) != 0;
  }
  uint64_t total;
  uint64_t pre = block_excl_scan_u64(local, scratch, &total);
  for (int b = b0; b < b1; ++b) {
    a.cbase[b] = pre;
    pre += a.part[b] & ~kNcBad;
  }
  bad = __syncthreads_or(bad) || total != uint64_t(a.n);
  if (threadIdx.x == 0) nc_verdict(a, bad);
}

__global__ void __launch_bounds__(kQThreads) k_nc_reduce(NcScanArgs a) {
  chain_begin();
  __shared__ uint64_t sh[kQThreads / 32];
  __shared__ int bad;
  if (threadIdx.x == 0) bad = 0;
  __syncthreads();
  const int64_t first = int64_t(blockIdx.x) * kQTile + int64_t(threadIdx.x) * kQItems;
  int32_t c[kQItems];
  load_counts(a.ncopies, a.n, first, c);
  if (a.clear_rs) {
    // the run-start array starts at -1 for the scan: this block's slice
    // [4096 b, 4096 b + 4096) of it, with 16-byte stores (the array is
    // 256-byte aligned) and single stores for a partial last vector
    int4* rs4 = reinterpret_cast<int4*>(a.runstart);
    const int64_t v0 = int64_t(blockIdx.x) * (kQTile / 4);
#pragma unroll
    for (int u = 0; u < kQTile / 4 / kQThreads; ++u) {
      const int64_t v = v0 + u * kQThreads + threadIdx.x;
      if (4 * v + 3 < a.n)
        rs4[v] = make_int4(-1, -1, -1, -1);
      else
        for (int64_t k = 4 * v; k < a.n; ++k) a.runstart[k] = -1;
    }
  }
  uint64_t s = 0;
  bool neg = false;
#pragma unroll
  for (int q = 0; q < kQItems; ++q) {
    neg |= c[q] < 0;
    s += uint64_t(uint32_t(max(c[q], 0)));
  }
  if (neg) bad = 1;
  s = warp_sum(s);
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    uint64_t t = 0;
    for (int w = 0; w < kQThreads / 32; ++w) t += sh[w];
    a.part[blockIdx.x] = t | (bad ? kNcBad : 0);
  }
  // (stamped calls: this block's share of the stamps, zero until the scan)
  const int stamps = kQTile >> src_shift(a.n);
  if (a.stamps && threadIdx.x < stamps && blockIdx.x * stamps + threadIdx.x < a.ntiles)
    a.stamps[blockIdx.x * stamps + threadIdx.x] = 0;
}

__global__ void __launch_bounds__(kFinThreads) k_nc_finalize(NcScanArgs a) { chain_begin(); nc_finalize_body(a); }

// Run starts of the block's items.  The block's outputs form the window
// [cbase, cbase + total); the windows of the blocks are disjoint and tile
// [0, n).  A window that fits shared memory is assembled there (-1, then the
// run starts) and written out with coalesced stores.  A larger one, when the
// run-start array holds -1 everywhere on entry (a sampler's, kept clean by
// the copy that consumes it), gets its run starts stored one by one.
// Stamped calls (a.stamps set; the stateless entry points, whose array is
// not cleared): every copy tile that receives a run start is stamped, and
// the copy reads the run starts of stamped tiles only, so a larger window
// sets -1 over all of itself when it has at most kFillAll rows, else over
// its part of its two edge copy tiles and of every copy tile where it puts a
// run start (over all of itself if those overflow a queue), before its run
// starts -- every slice the copy reads is then written in this call.
constexpr int kNcWin = 8192;
constexpr int kFillTiles = 1024;
constexpr uint64_t kFillAll = 1u << 17;

__global__ void __launch_bounds__(kQThreads) k_nc_scan(NcScanArgs a) {
  chain_begin();
  if (a.st->err) return;
  __shared__ __align__(16) int32_t win[kNcWin];
  __shared__ uint64_t scratch[33];
  __shared__ BigRuns big;
  __shared__ int s_nfill;
  // (a window is staged or its tiles are queued, never both)
  int64_t* const s_fill = reinterpret_cast<int64_t*>(win);
  static_assert(sizeof(win) >= kFillTiles * sizeof(int64_t), "the queue's space");
  const int sh = src_shift(a.n);
  __shared__ int s_has[kNcWin / kRTile + 2];  // staged window: its tiles that receive a run start
  if (threadIdx.x == 0) {
    big.count = 0;
    s_nfill = 0;
  }
  if (threadIdx.x < kNcWin / kRTile + 2) s_has[threadIdx.x] = 0;
  const int64_t n = a.n;
  const uint64_t un = uint64_t(n);
  const int64_t base = int64_t(blockIdx.x) * kQTile;
  const int64_t i0 = base + int64_t(threadIdx.x) * kQItems;
  int32_t c[kQItems];
  load_counts(a.ncopies, n, i0, c);
  uint64_t tsum = 0;
#pragma unroll
  for (int q = 0; q < kQItems; ++q) tsum += uint32_t(c[q]);
  uint64_t btot;
  const uint64_t w0 = a.cbase[blockIdx.x];
  const uint64_t excl = block_excl_scan_u64(tsum, scratch, &btot);  // (block barriers inside)
  const uint64_t wend = min(w0 + btot, un);
  const bool staged = btot <= uint64_t(kNcWin);
  const bool stamped = a.stamps != nullptr;
  const bool fill_all = stamped && !staged && btot <= kFillAll;
  int32_t* __restrict__ rsa = rs_now(a.runstart, a.runstart_alt, a.st);
  if (staged) {
    for (int k = threadIdx.x; k < int(btot); k += blockDim.x) win[k] = -1;
  } else if (stamped && !fill_all && threadIdx.x == 0 && w0 < wend) {
    s_fill[0] = int64_t(w0 >> sh);  // the edge tiles, shared with the neighbouring windows
    s_fill[1] = int64_t((wend - 1) >> sh);
    s_nfill = 2;
  }
  __syncthreads();
  uint64_t o = w0 + excl;
  if (stamped && !staged) {
    if (!fill_all) {
      int64_t last = -1;
#pragma unroll
      for (int q = 0; q < kQItems; ++q) {
        if (c[q] > 0 && i0 + q < n && o < un && int64_t(o >> sh) != last) {
          last = int64_t(o >> sh);
          const int slot = atomicAdd(&s_nfill, 1);
          if (slot < kFillTiles) s_fill[slot] = last;
        }
        o += uint32_t(c[q]);
      }
      __syncthreads();
    }
    if (fill_all || s_nfill > kFillTiles) {
      for (uint64_t k = w0 + threadIdx.x; k < wend; k += blockDim.x) rsa[k] = -1;
    } else {
      for (int f = 0; f < s_nfill; ++f) {
        const uint64_t t0 = max(w0, uint64_t(s_fill[f]) << sh);
        const uint64_t t1 = min(wend, (uint64_t(s_fill[f]) + 1) << sh);
        for (uint64_t k = t0 + threadIdx.x; k < t1; k += blockDim.x) rsa[k] = -1;
      }
    }
    __syncthreads();  // every -1 before any run start
    o = w0 + excl;
  }
  const uint64_t tfirst = w0 >> sh;
  int64_t stamped_tile = -1;  // (a thread's items are consecutive: one stamp per tile it reaches)
#pragma unroll
  for (int q = 0; q < kQItems; ++q) {
    const int64_t i = i0 + q;
    if (c[q] > 0 && i < n && o < un) {
      if (staged) {
        win[o - w0] = int32_t(i);
        if (stamped) s_has[(o >> sh) - tfirst] = 1;
      } else {
        rsa[o] = int32_t(i);
        if (stamped && int64_t(o >> sh) != stamped_tile) {
          stamped_tile = int64_t(o >> sh);
          a.stamps[stamped_tile] = 1;
        }
      }
      tile_starts_of_run(a.tile_src, o, o + uint32_t(c[q]), un, int32_t(i), big);
    }
    o += uint32_t(c[q]);
  }
  tile_starts_flush(a.tile_src, big);  // (block barrier inside)
  if (staged) {
    int32_t* __restrict__ rs = rsa + w0;
    for (int k = threadIdx.x; w0 + uint64_t(k) < wend; k += blockDim.x) rs[k] = win[k];
    if (stamped && threadIdx.x < kNcWin / kRTile + 2 && s_has[threadIdx.x]) a.stamps[tfirst + threadIdx.x] = 1;
  }
}

// Up to kNcSmall blocks of counts: the three passes as one.  Every block reads
// all counts (at most 512 KB from L2), so it knows its own prefix and the
// total without a launch before it, and writes its whole output window, so
// that no run start of an earlier call is left and no stamps are needed.
// (n = 65537: 13 us, against 16 in three launches and two memsets.)
constexpr int kNcSmall = 32;

__global__ void __launch_bounds__(kQThreads) k_nc_small(NcScanArgs a) {
  chain_begin();
  __shared__ int32_t win[kNcWin];
  __shared__ uint64_t scratch[33];
  __shared__ uint64_t sh[kQThreads / 32][2];
  __shared__ BigRuns big;
  const int64_t n = a.n;
  const uint64_t un = uint64_t(n);
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  if (threadIdx.x == 0) big.count = 0;
  int32_t c[kQItems];
  uint64_t before = 0, total = 0, tsum = 0;
  bool neg = false;
  // (the sums only need every count once: coalesced 16-byte loads, eight in
  // flight per thread; the block's own counts again, 16 per thread in order)
  load_counts(a.ncopies, n, int64_t(blockIdx.x) * kQTile + int64_t(threadIdx.x) * kQItems, c);
  const int64_t own = int64_t(blockIdx.x) * kQTile;
  auto add = [&](int32_t v, int64_t i) {
    neg |= v < 0;
    const uint32_t u = uint32_t(max(v, 0));
    total += u;
    if (i < own) before += u;
  };
  int64_t done = 0;
  if ((reinterpret_cast<uintptr_t>(a.ncopies) & 15) == 0) {
    const int4* p = reinterpret_cast<const int4*>(a.ncopies);
    const int n4 = int(n / 4);
    for (int e = threadIdx.x; e < n4; e += 8 * kQThreads) {
      int4 v[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const int k = e + u * kQThreads;
        v[u] = k < n4 ? __ldg(p + k) : make_int4(0, 0, 0, 0);
      }
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const int64_t i = 4 * int64_t(e + u * kQThreads);  // (a tile starts at a multiple of 4)
        neg |= (v[u].x | v[u].y | v[u].z | v[u].w) < 0;
        const uint64_t t = uint64_t(uint32_t(max(v[u].x, 0))) + uint32_t(max(v[u].y, 0)) + uint32_t(max(v[u].z, 0)) +
                           uint32_t(max(v[u].w, 0));
        total += t;
        if (i < own) before += t;
      }
    }
    done = 4 * int64_t(n4);
  }
  for (int64_t i = done + threadIdx.x; i < n; i += kQThreads) add(a.ncopies[i], i);
#pragma unroll
  for (int q = 0; q < kQItems; ++q) tsum += uint32_t(max(c[q], 0));
  before = warp_sum(before);
  total = warp_sum(total);
  if (lane == 0) {
    sh[wid][0] = before;
    sh[wid][1] = total;
  }
  neg = __syncthreads_or(neg);
  uint64_t w0 = 0;
  total = 0;
  for (int w = 0; w < kQThreads / 32; ++w) {
    w0 += sh[w][0];
    total += sh[w][1];
  }
  const bool bad = neg || total != un;
  if (blockIdx.x == 0 && threadIdx.x == 0) nc_verdict(a, bad);
  if (bad || (!a.reset_err && a.st->err)) return;
  uint64_t btot;
  const uint64_t excl = block_excl_scan_u64(tsum, scratch, &btot);
  const bool staged = btot <= uint64_t(kNcWin);
  int32_t* __restrict__ rs = rs_now(a.runstart, a.runstart_alt, a.st) + w0;
  if (staged) {
    for (int k = threadIdx.x; k < int(btot); k += blockDim.x) win[k] = -1;
  } else {
    for (uint64_t k = threadIdx.x; k < btot; k += blockDim.x) rs[k] = -1;
  }
  __syncthreads();  // every -1 before any run start
  uint64_t o = excl;
  const int64_t i0 = int64_t(blockIdx.x) * kQTile + int64_t(threadIdx.x) * kQItems;
#pragma unroll
  for (int q = 0; q < kQItems; ++q) {
    if (c[q] > 0) {
      if (staged)
        win[o] = int32_t(i0 + q);
      else
        rs[o] = int32_t(i0 + q);
      tile_starts_of_run(a.tile_src, w0 + o, w0 + o + uint32_t(c[q]), un, int32_t(i0 + q), big);
      o += uint32_t(c[q]);
    }
  }
  tile_starts_flush(a.tile_src, big);  // (block barrier inside)
  if (staged)
    for (int k = threadIdx.x; k < int(btot); k += blockDim.x) rs[k] = win[k];
}

// ---------------------------------------------------------------- redistribute
// Shared memory of one redistribute block, declared by the calling kernel so
// that kernels dispatching to several row sizes hold one copy.
template <int TILE>
struct RedistSmemT {
  int32_t mark[TILE];
  int32_t wsc[kRThreads / 32];
};
using RedistSmem = RedistSmemT<kCopyTile>;

// One tile of TILE output rows, which a source entry's rows divide.
template <typename V, int CPR, int KU = 8, bool COH = false, int TILE = kCopyTile>
__device__ __forceinline__ void redistribute_body(const RedistArgs& a, const int blk, RedistSmemT<TILE>& sm) {
  int cur = 0;
  if (a.stateful) {
    if (a.use_pending ? !a.st->pending : !(a.force || a.st->flag)) return;
    cur = a.st->cur;
  }
  // after an error nothing is copied, but the runstart slice is still reset
  const bool failed = a.st->err != 0;
  int32_t* const mark = sm.mark;
  int32_t* const wsc = sm.wsc;
  const int64_t n = a.n;
  const int64_t k0 = int64_t(blk) * TILE;
  const int len = int(n - k0 < TILE ? n - k0 : int64_t(TILE));
  // this tile's slice of runstart (survivor runs starting here), reset to -1
  // for the next resampling
  int32_t* __restrict__ rs = rs_now(a.runstart, a.runstart_alt, a.st) + k0;
  constexpr int kItems = TILE / kRThreads;
  static_assert(TILE % kRTile == 0 && kRTile % kRThreads == 0, "whole rounds of the block per source entry");
  const int sh = src_shift(n);
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  int32_t v[kItems];
#pragma unroll
  for (int u = 0; u < kItems; ++u) {
    const int k = threadIdx.x + u * kRThreads;
    // (a stamped stateless call: an unstamped entry's rows have no run starts,
    // and their slice is neither read nor reset)
    const bool read = !a.stamps || (k < len && a.stamps[(k0 + u * kRThreads) >> sh]);
    v[u] = (read && k < len) ? rs[k] : -1;
  }
  // the run covering the first output row may have started in an earlier tile
  const int32_t first =
      threadIdx.x == 0 ? min(max(a.tile_src[k0 >> sh], 0), int32_t(n - 1)) : -1;
#pragma unroll
  for (int u = 0; u < kItems; ++u) {
    const int k = threadIdx.x + u * kRThreads;
    // reset only the entries that were set (rewriting the whole slice was
    // measured slower); stamped calls need no reset
    if (!a.stamps && k < len && v[u] >= 0) rs[k] = -1;
    v[u] = v[u] < int32_t(n) ? v[u] : int32_t(n - 1);
  }
  v[0] = max(v[0], first);
  if (failed) return;
  // inclusive max-scan over the tile: kItems consecutive entries per thread
  // (one: straight from the register)
  int run = v[0];
  const int b = threadIdx.x * kItems;
  if constexpr (kItems > 1) {
#pragma unroll
    for (int u = 0; u < kItems; ++u) mark[threadIdx.x + u * kRThreads] = v[u];
    __syncthreads();
    run = -1;
#pragma unroll
    for (int q = 0; q < kItems; ++q) run = max(run, mark[b + q]);
  }
  {
    const int incl = warp_incl_max_i32(run);
    if (lane == 31) wsc[wid] = incl;
    __syncthreads();
    int carry = -1;
    for (int w = 0; w < wid; ++w) carry = max(carry, wsc[w]);
    if constexpr (kItems > 1) {
      int excl = __shfl_up_sync(0xffffffffu, incl, 1);
      if (lane == 0) excl = -1;
      run = max(carry, excl);
#pragma unroll
      for (int q = 0; q < kItems; ++q) {
        run = max(run, mark[b + q]);
        mark[b + q] = run;
      }
    } else {
      mark[threadIdx.x] = max(carry, incl);
    }
  }
  __syncthreads();
  // copy rows: element e of the tile is chunk (e % cpr) of row (e / cpr)
  const int cpr = CPR > 0 ? CPR : a.row_bytes / int(sizeof(V));
  const V* __restrict__ in = static_cast<const V*>(cur ? a.x_in[1] : a.x_in[0]);
  V* __restrict__ out = static_cast<V*>(cur ? a.x_out[1] : a.x_out[0]) + k0 * cpr;
  const int total = len * cpr;
  constexpr int kU = KU;  // loads in flight per thread
  for (int e0 = threadIdx.x; e0 < total; e0 += kRThreads * kU) {
    V v[kU];
#pragma unroll
    for (int u = 0; u < kU; ++u) {
      const int e = e0 + u * kRThreads;
      if (e < total) {
        const int k = e / cpr, c = e - k * cpr;
        v[u] = ld_rows<COH>(in + int64_t(mark[k]) * cpr + c);
      }
    }
#pragma unroll
    for (int u = 0; u < kU; ++u) {
      const int e = e0 + u * kRThreads;
      if (e < total) out[e] = v[u];
    }
  }
  if (a.lp_bytes == 4) {
    const uint32_t* __restrict__ li = static_cast<const uint32_t*>(cur ? a.lp_in[1] : a.lp_in[0]);
    uint32_t* __restrict__ lo = static_cast<uint32_t*>(cur ? a.lp_out[1] : a.lp_out[0]) + k0;
    for (int k = threadIdx.x; k < len; k += kRThreads) lo[k] = ld_plain<COH>(li + mark[k]);
  } else if (a.lp_bytes == 8) {
    const uint64_t* __restrict__ li = static_cast<const uint64_t*>(cur ? a.lp_in[1] : a.lp_in[0]);
    uint64_t* __restrict__ lo = static_cast<uint64_t*>(cur ? a.lp_out[1] : a.lp_out[0]) + k0;
    for (int k = threadIdx.x; k < len; k += kRThreads) lo[k] = ld_plain<COH>(li + mark[k]);
  }
  if (a.logw) {
    const double reset = a.stateful ? a.st->reset_logw : a.reset_logw;
    double* __restrict__ lw = a.logw + k0;
    for (int k = threadIdx.x; k < len; k += kRThreads) lw[k] = reset;
  }
}

template <typename V, int CPR, int TILE>
__global__ void __launch_bounds__(kRThreads) k_redistribute(RedistArgs a) {
  chain_begin();
  __shared__ RedistSmemT<TILE> sm;
  redistribute_body<V, CPR, 8, false, TILE>(a, blockIdx.x, sm);
  if (a.end_iter) end_iteration(a.st, gridDim.x, 0);
}

// ---------------------------------------------------------------- one-tile samplers
// A fused small sampler that also returns the covariance
// ends its last iteration with redistribute and commit as one kernel.
template <typename V>
__global__ void __launch_bounds__(kRThreads) k_redistribute_commit(RedistArgs a, int d, int force_flip, int recycle) {
  __shared__ RedistSmemT<kRTile> sm;
  redistribute_body<V, 0, 8, false, kRTile>(a, 0, sm);
  __syncthreads();
  if (threadIdx.x < 32) commit_warp(a.st, d, force_flip, recycle);
}

// ---------------------------------------------------------------- fused small-sampler iterations
// FP64 samplers of few particles and coordinates (see small_iter_fits): k
// iterations of Algorithm 2 in one cooperative launch.  Every block runs its
// share of the move + reweight with the particle-to-thread map of the
// separate move launch (move_threads per block own particles); then block 0
// alone runs, in the order of the separate launches, t += 1, the maximum, the
// quantise reduce / finalise / scan, the copy and the commit -- the bodies of
// k_max_finalize, k_quant_reduce / finalize / scan and k_redistribute_commit -- so the results
// are bit for bit those of the separate launches.  At this size an iteration
// is a chain of dependent FP64 operations (tens to thousands of cycles each
// on this GPU) and kernel boundaries; two grid barriers per iteration replace
// the five boundaries.
//
// The grid barrier (every block is resident: cooperative launch): one 64-bit
// count of arrivals, zeroed before the launch; a block's b-th barrier of the
// launch (b = 1, 2, ...) completes when the count reaches b (grid + extra).
// A block adds its arrival (release) and polls the count (acquire) -- for at
// most half a second of the global timer (and at most 2^24 polls), after
// which it records SMC_ETIMEOUT and the kernel returns.  extra: arrivals
// expected beyond the grid (0; 1 only in the stall test, where every wait
// runs out).
constexpr unsigned long long kBarrierNs = 500000000ull;
constexpr long long kBarrierPolls = 1ll << 24;

__device__ __forceinline__ unsigned long long ld_acquire_u64(const unsigned long long* p) {
  unsigned long long v;
  asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}

__device__ __forceinline__ void red_release_add_u64(unsigned long long* p, unsigned long long v) {
  asm volatile("red.release.gpu.global.add.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}

__device__ __forceinline__ unsigned long long global_ns() {
  unsigned long long v;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(v));
  return v;
}

__device__ __forceinline__ bool grid_barrier(unsigned long long* bar, unsigned long long& nbar, DevState* st,
                                             unsigned extra) {
  __shared__ int s_ok;
  ++nbar;
  __syncthreads();
  if (threadIdx.x == 0) {
    const unsigned long long target = nbar * (gridDim.x + extra);
    red_release_add_u64(bar, 1ull);
    int ok = 1;
    const unsigned long long t0 = global_ns();
    for (long long polls = 0; ld_acquire_u64(bar) < target; ++polls) {
      if (polls > kBarrierPolls || global_ns() - t0 > kBarrierNs) {
        record_error(st, SMC_ETIMEOUT);
        ok = 0;
        break;
      }
      __nanosleep(64);
    }
    __threadfence();
    s_ok = ok;
  }
  __syncthreads();
  return s_ok != 0;
}

// The stages' shared memory overlaps (each phase writes what it reads before
// reading it, and phases are separated by block barriers).
union SmallIterSmem {
  TargetSmem<double> ts;
  QuantReduceSmem q;
  ScanSmem sc;
  RedistSmemT<kRTile> r;
};

template <typename V>
__global__ void __launch_bounds__(kQThreads) k_iterate_small(SmallIterArgs s) {
  constexpr int DMAX = 4;  // (the separate kernels' width class)
  static_assert(kSmallIterD <= DMAX, "coordinates");
  __shared__ SmallIterSmem sm;
  TargetSmem<double>& ts = sm.ts;
  QuantReduceSmem& qsm = sm.q;
  RedistSmemT<kRTile>& rsm = sm.r;
  DevState* st = s.a.st;
  unsigned long long* const bar = s.bar;
  unsigned long long nbar = 0;
  const unsigned extra = s.stall ? 1u : 0u;
  for (int it = 0; it < s.k; ++it) {
    move_reweight_generic_body<double, DMAX, true, true>(s.a, ts, blockIdx.x, gridDim.x, s.move_threads, 1);
    if (!grid_barrier(bar, nbar, st, extra)) return;
    if (blockIdx.x == 0) {
      if (threadIdx.x == 0) st->t += 1;
      __syncthreads();
      max_finalize_body(s.a.part, gridDim.x, st);
      __syncthreads();
      quant_reduce_body<double, DMAX, true, true>(s.q, 0, qsm);
      __syncthreads();
      quant_finalize_body(s.q, 0);
      __syncthreads();
      if (s.a.n <= kQThreads)
        quant_scan_body<1>(s.q, 0, s.q.cbase[0], sm.sc);
      else
        quant_scan_body<2>(s.q, 0, s.q.cbase[0], sm.sc);
      if (!(s.stop_last && it + 1 == s.k)) {
        __syncthreads();
        redistribute_body<V, 0, 8, true, kRTile>(s.r, 0, rsm);
        __syncthreads();
        if (threadIdx.x < 32) commit_warp(st, s.d, 0, 1);
      }
    }
    if (it + 1 < s.k && !grid_barrier(bar, nbar, st, extra)) return;
  }
}

// Few particles with few coordinates, unless every iteration resamples: block
// 0 runs the stages one after another on its own, so it loses where they have
// work to share out.  Measured per iteration (fused, separate kernels, us):
//   D = 1  N = 64 21.8, 24.1   N = 256 22.4, 23.0   N = 512 24.1, 24.9
//   D = 2  N = 64 20.0, 21.0   N = 256 21.5, 21.6   N = 300 22.5, 23.1   N = 512 22.8, 22.8
//   D = 3  N = 64 23.1, 23.6   N = 256 25.4, 25.6   N = 300 26.1, 25.5
//   D = 4  N = 64 24.1, 23.3   N = 256 26.2, 26.1   N = 512 28.3, 26.1
//   D = 8  N = 64 36.6, 33.7   D = 32  N = 64 107.9, 102.0
// and with a copy in every iteration D = 1  N = 64 25.1, 23.9, D = 3  N = 256 27.6, 27.5.
static_assert(kSmallIter <= kRTile && kSmallIter <= 2 * kQThreads, "one copy tile, two scan items per thread");
bool small_iter_fits(int64_t n, int d, int dtype, int mode) {
  return dtype == SMC_F64 && mode != SMC_RESAMPLE_ALWAYS && n <= (d <= 2 ? kSmallIter : kSmallIter / 2) &&
         d <= kSmallIterD;
}

cudaError_t launch_iterate_small(const SmallIterArgs& s, int move_blocks, cudaStream_t st) {
  if (!small_iter_fits(s.a.n, s.d, s.a.dtype, s.q.mode) || s.k < 1 || move_blocks < 1 || s.move_threads < 1 ||
      s.move_threads > kQThreads || s.d < 1 || s.r.row_bytes % 8 != 0)
    return cudaErrorInvalidValue;
  SmallIterArgs a = s;
  void* args[] = {&a};
  const void* fn = (s.r.row_bytes % 16 == 0) ? reinterpret_cast<const void*>(&k_iterate_small<uint4>)
                                             : reinterpret_cast<const void*>(&k_iterate_small<uint2>);
  return cudaLaunchCooperativeKernel(fn, dim3(move_blocks), dim3(kQThreads), args, 0, st);
}

// ---------------------------------------------------------------- batched launches
// One launch per stage for many samplers: block b of the launch runs block
// map[b].y of sampler map[b].x with that sampler's own arguments, so every
// sampler's blocks, reductions and results are those of its own launch.
__device__ __forceinline__ int dclass(int d) { return d <= 4 ? 0 : (d <= 8 ? 1 : (d <= 16 ? 2 : 3)); }

// left (standing batches of slots; NULL otherwise): see k_move_reweight_batch.
// A slot's map covers its capacity; blocks past the member's own count exit.
// WIDE: members of D > 16 too.  Their route has 32 column sums and as many loaded
// values in registers (124 against 80 a thread), which costs the others a third
// of their resident warps: two members of 2^22, D = 16 125 against 101 us, D = 4 100
// against 85; six of 10^5, D = 32 31 with it, 42 before they had the route.
template <bool WIDE>
__global__ void __launch_bounds__(kQThreads) k_quant_reduce_batch(const QuantArgs* __restrict__ qa,
                                                                 const int4* __restrict__ map,
                                                                 const int32_t* __restrict__ left) {
  __shared__ QuantReduceSmem sm;
  const int4 m = map[blockIdx.x];
  if (left && left[m.x] <= 0) return;
  const QuantArgs a = qa[m.x];
  if (m.y >= a.nblocks) return;
  switch (dclass(a.d)) {
    case 0: quant_reduce_body<float, 4, true>(a, m.y, sm); break;
    case 1: quant_reduce_body<float, 8, true>(a, m.y, sm); break;
    case 2: quant_reduce_body<float, 16, true>(a, m.y, sm); break;
    default:
      if constexpr (WIDE) quant_reduce_body<float, 32, true>(a, m.y, sm);
      break;
  }
}

__global__ void __launch_bounds__(kFinBatchThreads) k_quant_finalize_batch(const QuantArgs* __restrict__ qa,
                                                                     const int32_t* __restrict__ left) {
  if (left && left[blockIdx.x] <= 0) return;
  const QuantArgs a = qa[blockIdx.x];
  quant_finalize_body(a, 0);
}

__global__ void __launch_bounds__(kQThreads, 4) k_quant_scan_batch(const QuantArgs* __restrict__ qa,
                                                               const int4* __restrict__ map,
                                                               const int32_t* __restrict__ left) {
  const int4 m = map[blockIdx.x];
  if (left && left[m.x] <= 0) return;
  const QuantArgs a = qa[m.x];
  if (m.y >= a.nblocks) return;
  __shared__ ScanSmem sm;
  quant_scan_body(a, int64_t(m.y) * kQTile, a.cbase[m.y], sm);
}

template <int KU>
__global__ void __launch_bounds__(kRThreads) k_redistribute_batch(const RedistArgs* __restrict__ ra,
                                                                 const int4* __restrict__ map,
                                                                 const int32_t* __restrict__ left) {
  __shared__ RedistSmem sm;
  const int4 m = map[blockIdx.x];
  if (left && left[m.x] <= 0) return;
  const RedistArgs a = ra[m.x];
  if (m.y >= a.ntiles) return;
  switch (a.row_bytes) {
    case 8: redistribute_body<uint2, 1, KU>(a, m.y, sm); break;
    case 16: redistribute_body<uint4, 1, KU>(a, m.y, sm); break;
    case 32: redistribute_body<uint4, 2, KU>(a, m.y, sm); break;
    case 64: redistribute_body<uint4, 4, KU>(a, m.y, sm); break;
    case 128: redistribute_body<uint4, 8, KU>(a, m.y, sm); break;
    default:
      if (a.row_bytes % 16 == 0)
        redistribute_body<uint4, 0, KU>(a, m.y, sm);
      else if (a.row_bytes % 8 == 0)
        redistribute_body<uint2, 0, KU>(a, m.y, sm);
      else
        redistribute_body<uint32_t, 0, KU>(a, m.y, sm);
      break;
  }
}

// Timing input for the copy stage: every tile's run starts set to the
// identity (each row its own single copy), which the copy consumes and resets
// to -1 as usual.
__global__ void __launch_bounds__(kRThreads) k_identity_runs_batch(const RedistArgs* __restrict__ ra,
                                                                  const int4* __restrict__ map) {
  const int4 m = map[blockIdx.x];
  const RedistArgs a = ra[m.x];
  const int64_t k0 = int64_t(m.y) * kCopyTile;
  const int len = int(a.n - k0 < kCopyTile ? a.n - k0 : int64_t(kCopyTile));
  int32_t* __restrict__ rs = rs_now(a.runstart, a.runstart_alt, a.st);
  const int sh = src_shift(a.n);
  for (int k = threadIdx.x; k < len; k += kRThreads) {
    rs[k0 + k] = int32_t(k0 + k);
    if ((k & ((1 << sh) - 1)) == 0) const_cast<int32_t*>(a.tile_src)[(k0 + k) >> sh] = int32_t(k0 + k);
  }
}

const void* quant_reduce_batch_kernel(bool wide) {
  return wide ? reinterpret_cast<const void*>(&k_quant_reduce_batch<true>)
              : reinterpret_cast<const void*>(&k_quant_reduce_batch<false>);
}
cudaError_t launch_quant_reduce_batch(const QuantArgs* qa, const int4* map, int nblocks, bool wide, cudaStream_t s,
                                      const int32_t* left) {
  (wide ? k_quant_reduce_batch<true> : k_quant_reduce_batch<false>)<<<nblocks, kQThreads, 0, s>>>(qa, map, left);
  return cudaGetLastError();
}
cudaError_t launch_quant_finalize_batch(const QuantArgs* qa, int count, cudaStream_t s, const int32_t* left) {
  k_quant_finalize_batch<<<count, kFinBatchThreads, 0, s>>>(qa, left);
  return cudaGetLastError();
}
cudaError_t launch_quant_scan_batch(const QuantArgs* qa, const int4* map, int nblocks, cudaStream_t s,
                                    const int32_t* left) {
  k_quant_scan_batch<<<nblocks, kQThreads, 0, s>>>(qa, map, left);
  return cudaGetLastError();
}
cudaError_t launch_redistribute_batch(const RedistArgs* ra, const int4* map, int nblocks, int copy_variant,
                                      cudaStream_t s, const int32_t* left) {
  switch (copy_variant) {
    case 0: k_redistribute_batch<4><<<nblocks, kRThreads, 0, s>>>(ra, map, left); break;
    case 1: k_redistribute_batch<8><<<nblocks, kRThreads, 0, s>>>(ra, map, left); break;
    case 2: k_redistribute_batch<16><<<nblocks, kRThreads, 0, s>>>(ra, map, left); break;
    default: return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}
cudaError_t launch_identity_runs_batch(const RedistArgs* ra, const int4* map, int nblocks, cudaStream_t s) {
  k_identity_runs_batch<<<nblocks, kRThreads, 0, s>>>(ra, map);
  return cudaGetLastError();
}

// ---------------------------------------------------------------- launchers
static int qblocks(int64_t n) { return int((n + kQTile - 1) / kQTile); }

cudaError_t launch_state_init(DevState* st, int64_t n, int64_t t, int F, cudaStream_t s) {
  chain_launch(k_state_init, 1, 32, 0, s, st, n, t, F);
  return cudaGetLastError();
}

cudaError_t launch_max_logw(const double* logw, int64_t n, DevState* st, cudaStream_t s) {
  chain_launch(k_max_logw, qblocks(n), kQThreads, 0, s, logw, n, st);
  return cudaGetLastError();
}

// Up to kQSplitTiles = 76 tiles of 4096 weights (their eighths are at most
// two blocks on each of 152 SMs): the cluster reduce and the scan of 512 items
// per block.  Measured (kernel, one block per tile -> eight): reduce at 5
// tiles, D = 32 41 -> 9.8 us; 64 tiles, D = 32 36 -> 20, FP64 D = 8 32 -> 21;
// 17 tiles without rows 15.6 -> 5.9, its scan 14.9 -> 5.5; but 245 tiles,
// D = 8 17 -> 28 and scan 13.0 -> 15.5 us, 4096 tiles 0.129 -> 0.50 ms (several
// waves of blocks that each wait for the weights, their cluster and shared
// memory of another SM).
static bool quant_split(int64_t n) { return qblocks(n) <= kQSplitTiles; }

template <typename ST>
static cudaError_t quant_reduce_t(const QuantArgs& a, cudaStream_t s) {
  const int g = qblocks(a.n);
  const bool est = a.x[0] && a.d >= 1;
  if (quant_split(a.n)) {
    if (!est)
      chain_launch(k_quant_reduce_cluster<ST, 1, false>, g * kQSplit, kQThreads, 0, s, a);
    else if (a.d <= 8)
      chain_launch(k_quant_reduce_cluster<ST, 1, true>, g * kQSplit, kQThreads, 0, s, a);
    else if (a.d <= 16)
      chain_launch(k_quant_reduce_cluster<ST, 2, true>, g * kQSplit, kQThreads, 0, s, a);
    else
      chain_launch(k_quant_reduce_cluster<ST, 4, true>, g * kQSplit, kQThreads, 0, s, a);
  } else if (!est) {
    chain_launch(k_quant_reduce<ST, 1, false>, g, kQThreads, 0, s, a);
  } else if (a.d <= 4) {
    chain_launch(k_quant_reduce<ST, 4, true>, g, kQThreads, 0, s, a);
  } else if (a.d <= 8) {
    chain_launch(k_quant_reduce<ST, 8, true>, g, kQThreads, 0, s, a);
  } else if (a.d <= 16) {
    chain_launch(k_quant_reduce<ST, 16, true>, g, kQThreads, 0, s, a);
  } else {
    chain_launch(k_quant_reduce<ST, 32, true>, g, kQThreads, 0, s, a);
  }
  return cudaGetLastError();
}

cudaError_t launch_quant_reduce(const QuantArgs& a, cudaStream_t s) {
  return a.dtype == SMC_F64 ? quant_reduce_t<double>(a, s) : quant_reduce_t<float>(a, s);
}

cudaError_t launch_quant_finalize(const QuantArgs& a, int set_lse_prev, cudaStream_t s) {
  k_quant_finalize<<<1, kFinThreads, 0, s>>>(a, set_lse_prev);
  return cudaGetLastError();
}

cudaError_t launch_quant_scan(const QuantArgs& a, cudaStream_t s) {
  if (quant_split(a.n))
    k_quant_scan_sub<<<qblocks(a.n) * kQSplit, kQThreads, 0, s>>>(a);
  else
    k_quant_scan<<<qblocks(a.n), kQThreads, 0, s>>>(a);
  return cudaGetLastError();
}

cudaError_t launch_iter_finalize(const QuantArgs& a, cudaStream_t s) {
  chain_launch(k_iter_finalize, 1, a.nblocks > 256 ? kFinThreads : 256, 0, s, a);
  return cudaGetLastError();
}

cudaError_t launch_iter_scan(const QuantArgs& a, cudaStream_t s) {
  if (quant_split(a.n))
    chain_launch(k_iter_scan<true>, qblocks(a.n) * kQSplit + 1, kQThreads, 0, s, a);
  else
    chain_launch(k_iter_scan<false>, qblocks(a.n) + 1, kQThreads, 0, s, a);
  return cudaGetLastError();
}

bool nc_small(int64_t n) { return qblocks(n) <= kNcSmall; }

cudaError_t launch_nc(const NcScanArgs& a, cudaStream_t s) {
  if (nc_small(a.n)) {
    chain_launch(k_nc_small, qblocks(a.n), kQThreads, 0, s, a);
    return cudaGetLastError();
  }
  chain_launch(k_nc_reduce, qblocks(a.n), kQThreads, 0, s, a);
  chain_launch(k_nc_finalize, 1, kFinThreads, 0, s, a);
  chain_launch(k_nc_scan, qblocks(a.n), kQThreads, 0, s, a);
  return cudaGetLastError();
}

template <int TILE>
static void redistribute_t(const RedistArgs& a, cudaStream_t s) {
  const int grid = int((a.n + TILE - 1) / TILE);
  const int rb = a.row_bytes;
  if (rb % 16 == 0) {
    switch (rb / 16) {
      case 1: chain_launch(k_redistribute<uint4, 1, TILE>, grid, kRThreads, 0, s, a); break;
      case 2: chain_launch(k_redistribute<uint4, 2, TILE>, grid, kRThreads, 0, s, a); break;
      case 4: chain_launch(k_redistribute<uint4, 4, TILE>, grid, kRThreads, 0, s, a); break;
      case 8: chain_launch(k_redistribute<uint4, 8, TILE>, grid, kRThreads, 0, s, a); break;
      default: chain_launch(k_redistribute<uint4, 0, TILE>, grid, kRThreads, 0, s, a); break;
    }
  } else if (rb % 8 == 0) {
    if (rb == 8)
      chain_launch(k_redistribute<uint2, 1, TILE>, grid, kRThreads, 0, s, a);
    else
      chain_launch(k_redistribute<uint2, 0, TILE>, grid, kRThreads, 0, s, a);
  } else {
    if (rb == 4)
      chain_launch(k_redistribute<uint32_t, 1, TILE>, grid, kRThreads, 0, s, a);
    else
      chain_launch(k_redistribute<uint32_t, 0, TILE>, grid, kRThreads, 0, s, a);
  }
}

cudaError_t launch_redistribute(const RedistArgs& a, cudaStream_t s) {
  // Up to kSmallCopy rows a block copies kRTile = 512 of them, above kCopyTile =
  // 1024.  A block's time is mostly latency (its run starts, the scan, the
  // gather), so a small copy needs many: 10 blocks of 2048 rows took 17.5 us
  // of an iteration at N = 20011, D = 32 (iteration 47.8 -> 41.6 us); a large one
  // fills the SMs either way and moves more bytes per block with 1024
  // (iteration at N = 2^24, D = 16 1.030 ms, with 512 1.046; at N = 2^20, D = 32
  // 0.171 and 0.169).
  if (a.n <= kSmallCopy)
    redistribute_t<kRTile>(a, s);
  else
    redistribute_t<kCopyTile>(a, s);
  return cudaGetLastError();
}

cudaError_t launch_redistribute_commit(const RedistArgs& a, int d, int force_flip, int recycle, cudaStream_t s) {
  if (a.n > kRTile || a.row_bytes % 8 != 0) return cudaErrorInvalidValue;
  if (a.row_bytes % 16 == 0)
    k_redistribute_commit<uint4><<<1, kRThreads, 0, s>>>(a, d, force_flip, recycle);
  else
    k_redistribute_commit<uint2><<<1, kRThreads, 0, s>>>(a, d, force_flip, recycle);
  return cudaGetLastError();
}

size_t devstate_bytes() { return sizeof(DevState); }

}  // namespace smc
