// k_moments.cu -- the weighted covariance beside the mean of eq. (7):
//
//   cov_ab = sum_i w~_i (x_ia - mean_a)(x_ib - mean_b),  w~_i = e^{log w_i - m} / s,
//
// a symmetric rank-N update of D(D+1)/2 sums.  A block stages a chunk of rows
// in shared memory (the centred row r and u = w r), then every thread
// advances a 4 x 4 tile of column pairs over its share of the chunk's rows
// (three 16-byte loads feed 16 pairs), with the sums in its registers for
// the whole launch.  The block's threads are (row group, tile): tiles of the
// upper triangle only, as many row groups as fit.
//
// What bounds it.  FP64 on this GPU runs at two lanes per SM and clock (FP32:
// 128), so products and sums of FP64 values set the pace whatever the
// memory does: the straightforward form of one FP64 multiply and one
// FP64 FMA per pair and row (plus two conversions, an exponential and a
// division per row) took 4.59 ms at N = 2^20, D = 32.  FP32 samplers
// therefore keep u and every sum as an unevaluated pair of FP32 values
// (error-free product by FMA, Knuth's two-sum: Dekker 1971; Knuth, TAOCP 2,
// 4.2.2), 11 FP32 operations per pair, and the weight comes from the integer
// exponential of the quantise pass with its exponent kept apart, so that a
// weight far below the largest keeps its relative precision.  The sums
// carry about 2^-45 relative error (with k rows per thread at most k^2 2^-48),
// far below the 2^-25 of rounding a row's
// difference to FP32 (the row precision), and no FP64 operation is left on
// the per-pair path.  FP64 samplers use FP64 FMAs, one per pair.  A block whose
// values or weights leave the range in which that holds (needs_fp64) is summed
// again in FP64.
//
// Measured (kernel alone): N = 2^20, D = 32 FP32 4.59 -> 0.33 ms (0.79 of the
// issue slots, 0.64 of the FP32 pipe); N = 2000003, D = 12 1.67 -> 0.165 ms.
// Packed two-lane FP32 instructions (27 % fewer instructions) were no faster
// (0.35 ms: the FP32 pipe does the same work).
#include <cmath>

#include "smc_internal.cuh"
#include "smc_kernels.h"

namespace smc {
namespace {

constexpr int kCovThreads = 256;
constexpr int kTileC = 4;  // a thread's tile: 4 x 4 column pairs

__host__ __device__ constexpr int cov_tiles(int nt) { return nt * (nt + 1) / 2; }

// A chunk holds at most kCap values per staged array (FP32: three arrays,
// FP64: two; below 48 KB) and 256 rows, a multiple of the row groups so that
// every thread has the same share.
template <typename T>
struct CovShape {
  static constexpr int kCap = sizeof(T) == 4 ? 3600 : 2048;
  static constexpr int kLoads = sizeof(T) == 4 ? 16 : 9;  // values a thread stages, at most (d = 20)
};

// index of tile t of the upper triangle of nt x nt tiles, row by row
__device__ __forceinline__ void tile_of(int t, int nt, int& ta, int& tb) {
  ta = 0;
  while (t >= nt - ta) {
    t -= nt - ta;
    ++ta;
  }
  tb = ta + t;
}

// e^{-a} = (h + l) 2^E, h in [1/2, 1], |l| < 2^-24, for finite |a| < 2048
// (larger: clamped; +inf is the caller's): the fixed-point exponential with a
// at 2^-53 and the exponent kept apart, about 2^-48 relative.
__device__ __forceinline__ void exp_split(double a, const uint64_t* __restrict__ T, float& h, float& l, int& E) {
  const uint64_t bits = (uint64_t)__double_as_longlong(a);
  const int e = min(int((bits >> 52) & 0x7ff), 1033);
  const uint64_t mant = (bits & 0x000FFFFFFFFFFFFFull) | (1ull << 52);
  const int sh = e - 1022;
  const uint64_t A = sh >= 0 ? (mant << sh) : (sh > -64 ? (mant >> (-sh)) : 0);
  const uint64_t L2E = 0x5C551D94AE0BF85Eull;  // round(log2(e) 2^62)
  const uint64_t zlo = A * L2E, zhi = __umul64hi(A, L2E);  // z = |a| log2(e) at 2^-115
  const int k = int(zhi >> 51);
  uint64_t f = (zhi << 13) | (zlo >> 51);
  E = -k;
  if (bits >> 63) {  // a < 0: 2^z = 2^(k + 1) 2^-(1 - f)
    E = f ? k + 1 : k;
    f = 0 - f;
  }
  const uint64_t M = exp2_neg_frac(f, T);  // ~2^62 2^-f
  h = float(uint32_t(M >> 38)) * 0x1p-24f;
  l = float(uint32_t(M >> 14) & 0xFFFFFFu) * 0x1p-48f;
}

// One pair and row of the FP32 path: (s, t) += (uh + ul) r.
__device__ __forceinline__ void pair_add(float uh, float ul, float r, float& s, float& t) {
  const float p = __fmul_rn(uh, r);
  const float e = __fmaf_rn(ul, r, __fmaf_rn(uh, r, -p));
  const float s1 = __fadd_rn(s, p);
  const float b = __fsub_rn(s1, s);
  const float d = __fadd_rn(__fsub_rn(s, __fsub_rn(s1, b)), __fsub_rn(p, b));
  t = __fadd_rn(t, __fadd_rn(d, e));
  s = s1;
}

// fl32(x - (mh + ml)), the difference formed with its rounding error.
__device__ __forceinline__ float centred(float x, float mh, float ml) {
  const float d = __fsub_rn(x, mh);
  const float b = __fsub_rn(d, x);
  const float e = __fsub_rn(__fsub_rn(x, __fsub_rn(d, b)), __fadd_rn(mh, b));
  return __fadd_rn(d, __fsub_rn(e, ml));
}

// The exponent of s (sums are kept at 2^-e of the weights e^{log w - m}, so that
// they reach no further than with w~ itself).
__device__ __forceinline__ int sum_exponent(double s) {
  const int e = (__double2hiint(s) >> 20) - 1023;
  return e > -1023 && e < 1024 ? e : 0;
}

// Whether a block's FP32 sums of a column may be off by more than 2^-36 of
// them, from the scaled column's largest |value| (its bits) and its sum of
// squares s.  Values stay below 2^40, so that no sum of 2^23 rows overflows.
// Weights below 2^-120 of the largest count as zero (at most 2^23 2^-120
// max^2), and additions below 2^-126 lose bits (2^23 2^-149 max).  Both are
// small against s unless the heavy rows' values are far below the largest one.
__device__ __forceinline__ bool needs_fp64(int max_bits, double s) {
  if (max_bits == 0) return false;
  const int R = (max_bits >> 23) - 126;  // max < 2^R
  if (R > 40) return true;
  const int least = max(2 * R - 61, max(R, 0) - 88);
  return !(s >= scalbn(1.0, least) && s < INFINITY);
}

// A block's sums in FP64, one pair per thread and turn: products and sums of
// FP64 values, the rows' differences rounded to FP32 as on the fast path.  FP64
// units bound it; only the blocks that need it come here (all of them at
// N = 2^20, D = 32: 4.7 ms beside the 0.33 of the fast path).
__device__ __noinline__ void block_fp64(const ParticleArgs& a, const float* __restrict__ x, int rows, double scale,
                                        float* s_r, double* s_w, double* __restrict__ out) {
  const int d = a.d, npairs = d * (d + 1) / 2, tid = threadIdx.x;
  const double m = a.st->m;
  const double* const mean = a.st->mean;
  constexpr int kPairs = (kMaxD * (kMaxD + 1) / 2 + kCovThreads - 1) / kCovThreads;
  double acc[kPairs] = {};
  int ca[kPairs], cb[kPairs];
  for (int k = 0; k < kPairs; ++k) {
    int p = min(tid + k * kCovThreads, npairs - 1);
    ca[k] = 0;
    while (p >= d - ca[k]) {
      p -= d - ca[k];
      ++ca[k];
    }
    cb[k] = ca[k] + p;
  }
  for (int64_t base = int64_t(blockIdx.x) * rows; base < a.n; base += int64_t(gridDim.x) * rows) {
    const int have = int(a.n - base < rows ? a.n - base : int64_t(rows));
    for (int e = tid; e < have * d; e += kCovThreads) s_r[e] = float(double(x[base * d + e]) - mean[e % d]);
    if (tid < have) {
      const double lw = a.logw[base + tid];
      s_w[tid] = lw == -INFINITY ? 0.0 : exp(lw - m) * scale;
    }
    __syncthreads();
    for (int k = 0; k < kPairs; ++k)
      if (tid + k * kCovThreads < npairs)
        for (int r = 0; r < have; ++r)
          acc[k] = fma(s_w[r] * double(s_r[r * d + ca[k]]), double(s_r[r * d + cb[k]]), acc[k]);
    __syncthreads();
  }
  for (int k = 0; k < kPairs; ++k)
    if (tid + k * kCovThreads < npairs) out[tid + k * kCovThreads] = acc[k];
}

// Partial sums covpart[block][pair] (pairs a <= b row by row).  The FP32
// path works on columns scaled by powers of two taken from the first rows
// (every block the same) and, in each block, on weights scaled by a running
// power of two.
template <typename T>
__global__ void __launch_bounds__(kCovThreads, 2) k_cov(ParticleArgs a, const double* cov,
                                                      double* __restrict__ covpart,
                                                      const uint64_t* __restrict__ exp_table) {
  chain_begin();
  using S = CovShape<T>;
  constexpr bool kF32 = sizeof(T) == 4;
  if (!cov) cov = a.st->cov_out;
  if (!cov || a.st->err) return;
  // r and u (FP32: u's low part too); afterwards the block's reduction space
  __shared__ __align__(16) T s_r[S::kCap];
  __shared__ __align__(16) T s_u[S::kCap];
  __shared__ __align__(16) T s_ul[kF32 ? S::kCap : 4];
  __shared__ float2 s_wf[kF32 ? kCovThreads : 1];
  __shared__ double s_wd[kF32 ? 1 : kCovThreads];
  __shared__ T s_mh[kMaxD], s_ml[kMaxD];
  __shared__ float s_inv[kMaxD];  // FP32: the columns' scale, a power of two
  __shared__ int s_ex[kMaxD];
  __shared__ uint64_t s_T[kF32 ? 128 : 1];
  __shared__ int s_emax[2];
  __shared__ int s_max[kF32 ? kMaxD : 1];  // FP32: the columns' largest |value| (scaled; its bits)
  __shared__ int s_redo;
  const int tid = threadIdx.x;
  const int d = a.d, nt = (d + kTileC - 1) / kTileC, nc = nt * kTileC;
  const int64_t n = a.n;
  const T* __restrict__ x = static_cast<const T*>(a.st->cur ? a.x[1] : a.x[0]);
  const double m = a.st->m;
  const int se = sum_exponent(a.st->est_s);
  const int tiles = cov_tiles(nt), groups = kCovThreads / tiles;
  const int rows = min(S::kCap / nc, kCovThreads) / groups * groups;
  // a thread stages one column's values of rows er, er + sr, ... (the first
  // sr d threads; coalesced)
  const int sr = kCovThreads / d, er = tid / d, ec = tid - er * d;
  const bool stages = er < sr;
  if (tid < kMaxD) {
    const double mu = tid < d ? a.st->mean[tid] : 0.0;
    s_mh[tid] = T(mu);
    s_ml[tid] = T(mu - double(T(mu)));
    s_ex[tid] = 0;
    if (kF32) s_max[tid] = 0;
  }
  if (tid == 0) s_redo = 0;
  if (kF32 && tid < 128) s_T[tid] = exp_table[tid];
  if (tid < 2) s_emax[tid] = -(1 << 20);
  for (int k = tid; k < S::kCap; k += kCovThreads) {  // (columns d .. nc stay zero)
    s_r[k] = T(0);
    s_u[k] = T(0);
    if (kF32) s_ul[k] = T(0);
  }
  __syncthreads();
  if constexpr (kF32) {
    // column scales: the exponent of the largest difference in the first rows
    for (int e = tid; e < min(n, int64_t(64)) * d; e += kCovThreads) {
      const int c = e % d;
      const float v = fabsf(centred(x[e], s_mh[c], s_ml[c]));
      if (v > 0.0f && v < INFINITY) atomicMax(&s_ex[c], (__float_as_int(v) >> 23) + 1);
    }
    __syncthreads();
    if (tid < kMaxD) {
      // r 2^-ex in about [0, 1]; both powers stay normal
      const int ex = s_ex[tid] ? max(-100, min(100, s_ex[tid] - 127)) : 0;
      s_ex[tid] = ex;
      s_inv[tid] = __int_as_float((127 - ex) << 23);
    }
    __syncthreads();
  }
  const int tile = tid % tiles, group = tid / tiles;
  int ta, tb;
  tile_of(tile, nt, ta, tb);
  T acc[kTileC * kTileC], low[kF32 ? kTileC * kTileC : 1];  // the sums (FP32: and their low parts)
#pragma unroll
  for (int k = 0; k < kTileC * kTileC; ++k) {
    acc[k] = T(0);
    if (kF32) low[k] = T(0);
  }
  T mh = T(0), ml = T(0);
  float inv = 1.0f;
  if (stages) {
    mh = s_mh[ec];
    ml = s_ml[ec];
    if (kF32) inv = s_inv[ec];
  }
  int K = -(1 << 20);  // FP32: weights are scaled by 2^-K
  int vmax = 0;        // FP32: the largest |value| this thread staged (its bits)
  const double scale = scalbn(1.0, -se);
  int turn = 0;
  // a chunk's values and log-weights are loaded while the one before it is
  // summed
  T v[S::kLoads];
  double lw = -INFINITY;
  auto load = [&](int64_t b) {
    const int have = int(max(int64_t(0), min(n - b, int64_t(rows))));
    const T* __restrict__ xb = x + b * d;
#pragma unroll
    for (int q = 0; q < S::kLoads; ++q) {
      const int r = er + q * sr;
      v[q] = (stages && r < have) ? xb[r * d + ec] : T(0);
    }
    lw = tid < have ? a.logw[b + tid] : -INFINITY;
  };
  load(int64_t(blockIdx.x) * rows);
  for (int64_t base = int64_t(blockIdx.x) * rows; base < n; base += int64_t(gridDim.x) * rows, turn ^= 1) {
    const int have = int(n - base < rows ? n - base : int64_t(rows));  // rows of this chunk
    if constexpr (kF32) {
      float h = 0.0f, l = 0.0f;
      int E = -(1 << 20);
      if (lw != -INFINITY) {
        const double a_i = m - lw;
        if (a_i > -INFINITY) {
          exp_split(a_i, s_T, h, l, E);
        } else {  // e^{inf} or NaN (log w is NaN or +inf, which the reweight reports): what it makes of the sums
          h = a_i == -INFINITY ? INFINITY : NAN;
          E = 0;
        }
      }
      const int em = __reduce_max_sync(0xffffffffu, E);
      if ((tid & 31) == 0) atomicMax(&s_emax[turn], em);
      __syncthreads();
      const int Kn = max(K, s_emax[turn]);
      if (tid == 0) s_emax[turn ^ 1] = -(1 << 20);
      if (Kn > K) {  // a larger weight than any before: the sums move to its scale
        const float f = Kn - K > 120 ? 0.0f : __int_as_float((127 - (Kn - K)) << 23);
#pragma unroll
        for (int k = 0; k < kTileC * kTileC; ++k) {
          acc[k] *= f;
          low[k] *= f;
        }
        K = Kn;
      }
      const float f = K - E > 120 ? 0.0f : __int_as_float((127 - (K - E)) << 23);
      s_wf[tid] = make_float2(h * f, l * f);
    } else {
      s_wd[tid] = lw == -INFINITY ? 0.0 : exp(lw - m) * scale;
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < S::kLoads; ++q) {
      const int r = er + q * sr;
      if (stages && r < rows) {
        const int at = r * nc + ec;
        if constexpr (kF32) {
          const float2 w = s_wf[r];
          const float rv = r < have ? centred(v[q], mh, ml) * inv : 0.0f;
          const float u = __fmul_rn(w.x, rv);
          vmax = max(vmax, __float_as_int(rv) & 0x7fffffff);
          s_r[at] = rv;
          s_u[at] = u;
          s_ul[at] = __fmaf_rn(w.y, rv, __fmaf_rn(w.x, rv, -u));
        } else {
          const double rv = r < have ? v[q] - mh : 0.0;
          s_r[at] = rv;
          s_u[at] = s_wd[r] * rv;
        }
      }
    }
    __syncthreads();
    load(base + int64_t(gridDim.x) * rows);
    if (group < groups) {
#pragma unroll 1
      for (int j = group; j < rows; j += groups) {
        const T* const pu = s_u + j * nc + ta * kTileC;
        const T* const pr = s_r + j * nc + tb * kTileC;
        if constexpr (kF32) {
          const float4 uh = *reinterpret_cast<const float4*>(pu);
          const float4 ul = *reinterpret_cast<const float4*>(s_ul + j * nc + ta * kTileC);
          const float4 rv = *reinterpret_cast<const float4*>(pr);
          const float uhv[4] = {uh.x, uh.y, uh.z, uh.w}, ulv[4] = {ul.x, ul.y, ul.z, ul.w};
          const float rvv[4] = {rv.x, rv.y, rv.z, rv.w};
#pragma unroll
          for (int p = 0; p < kTileC; ++p)
#pragma unroll
            for (int q = 0; q < kTileC; ++q)
              pair_add(uhv[p], ulv[p], rvv[q], acc[p * kTileC + q], low[p * kTileC + q]);
        } else {
          double u[kTileC], rr[kTileC];
#pragma unroll
          for (int p = 0; p < kTileC; ++p) {
            u[p] = pu[p];
            rr[p] = pr[p];
          }
          if (nt > 1) {
#pragma unroll
            for (int p = 0; p < kTileC; ++p)
#pragma unroll
              for (int q = 0; q < kTileC; ++q) acc[p * kTileC + q] = fma(u[p], rr[q], acc[p * kTileC + q]);
          } else {  // one tile: the pairs it does not need are skipped by all threads alike
#pragma unroll
            for (int p = 0; p < kTileC; ++p)
#pragma unroll
              for (int q = p; q < kTileC; ++q)
                if (q < d) acc[p * kTileC + q] = fma(u[p], rr[q], acc[p * kTileC + q]);
          }
        }
      }
    }
    __syncthreads();
  }
  // the row groups' sums, one row of every tile at a time through the space
  // of the staged rows: `per` threads for each sum (as many as the block
  // has, at most a warp) add every per-th group in order, then a fixed tree
  double* const red = reinterpret_cast<double*>(s_r);  // groups x tiles x 4 doubles
  static_assert(sizeof(s_r) >= size_t(kCovThreads) * kTileC * sizeof(double), "reduction space");
  const int npairs = d * (d + 1) / 2;
  double* const out = covpart + size_t(blockIdx.x) * npairs;
  if (kF32 && vmax) atomicMax(&s_max[ec], vmax);  // (seen behind the barriers below)
  int per = 32;
  while (per * tiles * kTileC > kCovThreads) per /= 2;
#pragma unroll
  for (int p = 0; p < kTileC; ++p) {
    if (group < groups) {
#pragma unroll
      for (int q = 0; q < kTileC; ++q)
        red[tid * kTileC + q] = kF32 ? double(acc[p * kTileC + q]) + double(low[kF32 ? p * kTileC + q : 0])
                                     : double(acc[p * kTileC + q]);
    }
    __syncthreads();
    const int k = tid / per, sub = tid % per;
    double s = 0.0;
    if (k < tiles * kTileC)
      for (int g = sub; g < groups; g += per) s += red[g * tiles * kTileC + k];
    for (int o = per / 2; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (k < tiles * kTileC && sub == 0) {
      int ra, rb;
      tile_of(k / kTileC, nt, ra, rb);
      const int ca = ra * kTileC + p, cb = rb * kTileC + k % kTileC;
      if (ca <= cb && cb < d) {
        if constexpr (kF32) {
          if (ca == cb && needs_fp64(s_max[ca], K > -(1 << 20) ? s : 1.0)) s_redo = 1;
          s = scalbn(s, K + s_ex[ca] + s_ex[cb] - se);
        }
        out[ca * d - ca * (ca - 1) / 2 + (cb - ca)] = s;
      }
    }
    __syncthreads();
  }
  if constexpr (kF32)
    if (s_redo) block_fp64(a, x, rows, scale, s_r, reinterpret_cast<double*>(s_wf), out);
}

// Sums the per-block partials, one warp per pair (lane l adds blocks l,
// l + 32, ... in order, then a fixed tree), divides by s and fills both
// triangles.  (One thread per pair walked up to 304 partials one FP64
// addition after another: 42 us.)
__global__ void __launch_bounds__(128) k_cov_finalize(const DevState* st, double* cov,
                                                     const double* __restrict__ covpart, int nblocks, int d) {
  chain_begin();
  if (!cov) cov = st->cov_out;
  if (!cov || st->err) return;
  const int npairs = d * (d + 1) / 2;
  const int p = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
  if (p >= npairs) return;
  double v = 0.0;
  for (int b = lane; b < nblocks; b += 32) v += covpart[size_t(b) * npairs + p];
  v = warp_sum(v);
  if (lane) return;
  v /= scalbn(st->est_s, -sum_exponent(st->est_s));
  int ca = 0, k = p;
  while (k >= d - ca) {
    k -= d - ca;
    ++ca;
  }
  const int cb = ca + k;
  cov[ca * d + cb] = v;
  cov[cb * d + ca] = v;
}

}  // namespace

cudaError_t launch_cov(const ParticleArgs& a, double* cov, double* covpart, int grid, cudaStream_t s) {
  const uint64_t* table = nullptr;
  cudaError_t e = expfx_table(&table);
  if (e != cudaSuccess) return e;
  if (a.dtype == SMC_F64)
    chain_launch(k_cov<double>, grid, kCovThreads, 0, s, a, cov, covpart, table);
  else
    chain_launch(k_cov<float>, grid, kCovThreads, 0, s, a, cov, covpart, table);
  e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  const int npairs = a.d * (a.d + 1) / 2;
  chain_launch(k_cov_finalize, (npairs + 3) / 4, 128, 0, s, a.st, cov, covpart, grid, a.d);
  return cudaGetLastError();
}

}  // namespace smc
