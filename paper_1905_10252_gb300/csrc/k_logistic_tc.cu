// k_logistic_tc.cu -- the Bayesian logistic-regression log-likelihood of every
// particle on the 5th-generation tensor cores (sm_103a), fused with the
// importance reweighting of eq. (5):
//
//   log pi(b) = b . v - sum_m softplus(z_m) - |b|^2 / (2 prior_var),
//   z = X b,  v = X^T y  (so sum_m y_m z_m = b . v needs no per-row work).
//
// Contraction.  A CTA takes two tiles of 128 particles (MMA M = 128) at a
// time and streams the data matrix past them through shared memory in half
// tiles of 128 rows (MMA N = 128, K = 32 features, zero padded).  FP32
// accuracy from BF16 tensor cores by the split x = hi + lo (hi = bf16(x),
// lo = bf16(x - hi)) on both operands:
//   z ~= B_hi X_hi + B_lo X_hi + B_hi X_lo   (FP32 accumulation in TMEM),
// dropping only B_lo X_lo (relative size 2^-16 of the product).
//
// Epilogue (one transcendental per matrix element).  The data
// images hold X log2(e), so the accumulator holds z' = z log2 e and, with
// a = |z'|:  softplus(z) = (z + a ln 2) / 2 + ln(1 + 2^-a), so
//   sum_m softplus(z_m) = (b . w + ln 2 sum_m a_m) / 2 + ln 2 sum_m log2(1 + e_m),
// w = column sums of X (FP64, once), e_m = ex2.approx(-a_m) on the
// multi-function unit (three instructions per element: |.| accumulate, ex2,
// product); the log2 is taken once per 16 rows of a running FP32
// product prod(1 + e_m) (each factor in (1, 2], so the product stays below
// 2^16).  Zero padding rows give z = 0 exactly and contribute exactly 1 to the
// log2 sum, removed as (m_pad - m).
//
// What bounds it.  ex2 runs at 32 lanes per SM and clock on this GPU (lg2 and
// the other functions at 16), so the epilogue's floor is 28 elements per SM
// and clock; the loop below alone, from TMEM, reaches 24.5, and the three
// MMAs of a product would allow about 42.  One tile of 128 particles per pass
// with 256-row MMAs, a wait for each tile before its first column is read,
// descriptors built and the abort flag read before every MMA ran at 13.6: a
// time line showed the issuing thread busy for 1900 cycles per 32768
// elements (530 of them for six MMAs, 160 for each wait of a phase long
// complete) and the epilogue waiting.  Two particle tiles share each half
// tile of data (half the L2 traffic, and one tile's MMAs run while the other's
// columns are read), descriptors advance by constants, completed phases cost
// one try_wait, each warp has its next 16 columns on the way across half
// tiles, and the loop holds no FP64 instruction (2 lanes per SM and clock;
// the flush of the sums to FP64 took a sixth of the time): sums of up to 8
// data tiles are added up as pairs of FP32 values (two-sum).
// N = 2^18, M = 8192, D = 32: 0.500 -> 0.394 ms, 13.6 -> 18.4 elements per SM
// and clock.
//
// Warp roles (20 warps): warp 0 lane 0 issues the bulk copies of the half
// tiles (8-stage ring, mbarrier complete_tx); warp 1 owns the TMEM allocation
// (512 columns: two 128 x 128 FP32 accumulators for each of the two particle
// tiles) and lane 0 issues the MMAs; warps 2-3 stage the particle tiles'
// BF16 hi / lo images (double buffered, so the next pair is staged while the
// current one is contracted); warps 4-19 run the epilogue, eight per
// particle tile: two per TMEM lane quarter, 64 columns each.
// Every
// mbarrier wait is bounded: on a timeout the CTA records SMC_ETIMEOUT, every
// role drains its remaining loop iterations without waiting (so the named
// barriers still match), waits (bounded) for its own copies in flight, frees
// TMEM and returns.
#include <atomic>

#include "smc_internal.cuh"
#include "smc_kernels.h"

namespace smc {
namespace {

constexpr int kTcPT = 128;                                  // particles per tile
constexpr int kTcPair = 2;                                  // particle tiles per pass over the data
constexpr int kTcRows = 128;                                // data rows per MMA (half an image tile)
constexpr int kTcStages = 8;                                // half tile ring
constexpr int kTcWarps = 20;
constexpr int kTcThreads = 32 * kTcWarps;
constexpr int kTcStageThreads = 64;                         // warps 2..3
constexpr int kTcEpiWarps = 16;                             // warps 4..19
constexpr int kTcTileThreads = 32 * kTcEpiWarps / kTcPair;  // epilogue threads of one particle tile
constexpr uint32_t kTcCols = 512;                           // TMEM columns
constexpr size_t kTcAImg = size_t(kTcPT) * kLgK * 2;        // one BF16 A image (8 KB)
constexpr size_t kTcBImg = size_t(kTcRows) * kLgK * 2;      // one BF16 image of a half tile (8 KB)
constexpr size_t kTcStageBytes = 2 * kTcBImg;               // hi | lo
constexpr int kTcPreRing = 4;                               // passes of per-particle constant terms in flight
// data ring + two pairs of (hi, lo) A images + the four sums per particle of
// the odd column groups + the ring of constant terms + barriers / TMEM slot /
// flags / warp maxima (1 KB) + alignment slack
constexpr size_t kTcSmem = kTcStages * kTcStageBytes + 2 * kTcPair * 2 * kTcAImg +
                           (4 + kTcPreRing) * kTcPair * kTcPT * sizeof(double) + 1024 + 1024;
constexpr long long kWaitCycles = 1ll << 31;                // ~1 s at 2 GHz

__device__ __forceinline__ uint32_t su32(const void* p) { return uint32_t(__cvta_generic_to_shared(p)); }

// tcgen05 shared-memory matrix descriptor: K-major, no swizzle; LBO = byte
// distance between core matrices adjacent in K, SBO = between 8-row groups.
__device__ __forceinline__ uint64_t mat_desc(uint32_t saddr, uint32_t lbo, uint32_t sbo) {
  return uint64_t((saddr >> 4) & 0x3FFF) | (uint64_t((lbo >> 4) & 0x3FFF) << 16) |
         (uint64_t((sbo >> 4) & 0x3FFF) << 32) | (uint64_t(1) << 46);
}

// kind::f16 instruction descriptor: FP32 accumulator, BF16 A and B, both
// K-major, N = 128, M = 128.
constexpr uint32_t kIdesc =
    (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t(kTcRows) >> 3) << 17) | ((uint32_t(kTcPT) >> 4) << 24);

__device__ __forceinline__ void mbar_init(uint64_t* b, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(su32(b)), "r"(count) : "memory");
}
__device__ __forceinline__ bool mbar_try(uint64_t* b, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(ok)
      : "r"(su32(b)), "r"(parity)
      : "memory");
  return ok != 0;
}
// Bounded wait; false after ~1 s (or at once when the phase is open and the
// CTA is already aborting; a complete phase is taken without a look at the flag).
__device__ __forceinline__ bool mbar_wait(uint64_t* b, uint32_t parity, volatile int* abort_flag) {
  if (mbar_try(b, parity)) return true;
  if (*abort_flag) return false;
  const long long t0 = clock64();
  while (!mbar_try(b, parity)) {
    if (*abort_flag) return false;
    if (clock64() - t0 > kWaitCycles) {
      *abort_flag = 1;
      return false;
    }
  }
  return true;
}
// The same for a whole warp, with one outcome for all lanes.  A phase that has
// completed is taken without a look at the abort flag (its data is valid).
__device__ __forceinline__ bool mbar_wait_warp(uint64_t* b, uint32_t parity, volatile int* abort_flag) {
  if (__all_sync(0xffffffffu, mbar_try(b, parity))) return true;
  return __all_sync(0xffffffffu, mbar_wait(b, parity, abort_flag));
}
__device__ __forceinline__ void mbar_arrive(uint64_t* b) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(su32(b)) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t* b, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(su32(b)), "r"(bytes) : "memory");
}
__device__ __forceinline__ void bulk_g2s(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                   su32(dst)),
               "l"(src), "r"(bytes), "r"(su32(bar))
               : "memory");
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void named_sync(int id, int threads) {
  asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(threads) : "memory");
}
template <int kAccumulate>
__device__ __forceinline__ void mma_bf16(uint32_t tmem_d, uint64_t da, uint64_t db) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
      " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem_d),
      "l"(da), "l"(db), "r"(kIdesc), "n"(kAccumulate)
      : "memory");
}
// One lane of the (converged) warp, the same at every call.
__device__ __forceinline__ bool elect_one() {
  uint32_t ok;
  asm volatile("{\n .reg .pred p;\n elect.sync _|p, 0xFFFFFFFF;\n selp.u32 %0, 1, 0, p;\n}\n" : "=r"(ok));
  return ok != 0;
}
__device__ __forceinline__ void mma_commit(uint64_t* bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(su32(bar))
               : "memory");
}
// 16 columns of the warp's lane quarter; complete after tmem_wait_ld.
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];\n"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr));
}
// The registers of a load pass through the wait, so that no use of them can
// be scheduled before it.
__device__ __forceinline__ void tmem_wait_ld(uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.wait::ld.sync.aligned;"
      : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]), "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]), "+r"(r[15])::"memory");
}
__device__ __forceinline__ float ex2_approx(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float lg2_approx(float x) {
  float y;
  asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ uint16_t bf16_rn(float f) {
  const uint32_t u = __float_as_uint(f);
  return uint16_t((u + 0x7FFFu + ((u >> 16) & 1u)) >> 16);
}
// byte offset of element (row r, column k) in a K-major core-matrix image
__device__ __forceinline__ uint32_t img_off(int r, int k) {
  return uint32_t((r >> 3) * 512 + (k >> 3) * 128 + (r & 7) * 16 + (k & 7) * 2);
}

// FP64 value of an FP32 number by its bits (no conversion instruction, which
// would take a slot of the FP64 pipe); zeros, subnormals, infinities and NaN
// (exponent field 0 or 255) are converted.  (The GPU's own NaN, 0x7FFFFFFF,
// rounds to -0 in the BF16 images: this is the way on which it reaches log pi.)
__device__ __forceinline__ double widen(float f) {
  const uint32_t u = __float_as_uint(f);
  if (((u + 0x00800000u) & 0x7F000000u) == 0) return double(f);
  return __hiloint2double(int((u & 0x80000000u) | (((u & 0x7FFFFFFFu) >> 3) + 0x38000000u)), int(u << 29));
}

// (hi, lo) += v: two-sum, so hi's rounding error is exact; only the additions
// of those errors into lo round (2^-24 of 2^-24 of the sum).
__device__ __forceinline__ void add_pair(float v, float& hi, float& lo) {
  const float s = __fadd_rn(hi, v);
  const float b = __fsub_rn(s, hi);
  lo = __fadd_rn(lo, __fadd_rn(__fsub_rn(hi, __fsub_rn(s, b)), __fsub_rn(v, b)));
  hi = s;
}
// The FP64 value of such a sum.  An infinite hi stands alone: the two-sum's
// error is then inf - inf.
__device__ __forceinline__ double pair_value(float hi, float lo) {
  return isinf(hi) ? double(hi) : double(hi) + double(lo);
}
// The sums of |z| are kept at this scale, so that a total of finite partial
// sums (2^20 of them at most: M < 2^31) stays finite, as it did in FP64.
constexpr float kAbsScale = 0x1p-24f;

__global__ void __launch_bounds__(kTcThreads, 1) k_logistic_tc(ParticleArgs a) {
  chain_begin();
  extern __shared__ uint8_t smem_raw[];
  uint8_t* sm = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t* xs = sm;                                   // kTcStages x (hi | lo) half tiles
  uint8_t* aimg = xs + kTcStages * kTcStageBytes;     // [2 buffers][kTcPair] x (hi, lo) particle tile images
  // [kTcPair][128][4]: |z| and log2 sums of the column groups 1 and 3
  double* s_part = reinterpret_cast<double*>(aimg + 2 * kTcPair * 2 * kTcAImg);
  // [kTcPreRing][kTcPair][128]: per particle b.(v - w / 2) - |b|^2 / (2 prior_var), a
  // ring of passes written by the stager warps
  double* s_pre = s_part + kTcPair * kTcPT * 4;
  uint64_t* full = reinterpret_cast<uint64_t*>(s_pre + kTcPreRing * kTcPair * kTcPT);
  uint64_t* empty = full + kTcStages;
  uint64_t* tfull = empty + kTcStages;   // [kTcPair][2]
  uint64_t* tempty = tfull + 2 * kTcPair;
  uint64_t* afull = tempty + 2 * kTcPair;
  uint64_t* aempty = afull + 2;
  uint64_t* prefull = aempty + 2;  // [kTcPreRing]
  uint32_t* tslot = reinterpret_cast<uint32_t*>(prefull + kTcPreRing);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tslot + 1);
  long long* wmax = reinterpret_cast<long long*>(tslot + 4);  // [kTcWarps]
  int* wnan = reinterpret_cast<int*>(wmax + kTcWarps);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const TargetDev* __restrict__ tg = a.tg;
  const int cur = a.st->cur;
  const float* __restrict__ x = static_cast<const float*>(cur ? a.x[1] : a.x[0]);
  float* __restrict__ lp = static_cast<float*>(cur ? a.logpi[1] : a.logpi[0]);
  const int64_t n = a.n;
  const int d = a.d;
  const int nx = tg->m_pad / kLgRows;  // image tiles, two half tiles each
  // this CTA's particle tiles, a contiguous share, two at a time
  const int64_t npt = (n + kTcPT - 1) / kTcPT;
  const int64_t pt0 = npt * blockIdx.x / gridDim.x, pt1 = npt * (blockIdx.x + 1) / gridDim.x;

  if (threadIdx.x == 0) {
    for (int s = 0; s < kTcStages; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    for (int b = 0; b < 2 * kTcPair; ++b) {
      mbar_init(&tfull[b], 1);
      mbar_init(&tempty[b], kTcEpiWarps / kTcPair);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&afull[b], kTcStageThreads);
      mbar_init(&aempty[b], 1);
    }
    for (int r = 0; r < kTcPreRing; ++r) mbar_init(&prefull[r], kTcStageThreads);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(su32(tslot)),
                 "r"(kTcCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tslot;

  MaxTracker mt;
  mt.init();

  if (warp == 0) {
    // ------------------------------------------------------------ producer
    if (lane == 0) {
      uint32_t g = 0, issued = 0, parity = 0;  // bit s: stage s was filled, and its last phase
      const uint8_t* img = reinterpret_cast<const uint8_t*>(tg->ximg);
      for (int64_t pt = pt0; pt < pt1; pt += kTcPair) {
        for (int j = 0; j < 2 * nx; ++j, ++g) {
          if (a.flags & PA_STALL_COPIES) continue;  // test hook: the consumers' waits run out
          const int s = int(g % kTcStages);
          const uint32_t r = g / kTcStages;
          if (!mbar_wait(&empty[s], (r & 1) ^ 1, abort_flag)) continue;
          mbar_expect_tx(&full[s], uint32_t(kTcStageBytes));
          // rows 128 (j & 1) .. of image tile j / 2: a run of its hi half and one of its lo half
          const uint8_t* src = img + size_t(j >> 1) * kLgTileBytes + size_t(j & 1) * kTcBImg;
          uint8_t* dst = xs + size_t(s) * kTcStageBytes;
          bulk_g2s(dst, src, uint32_t(kTcBImg), &full[s]);
          bulk_g2s(dst + kTcBImg, src + kLgTileBytes / 2, uint32_t(kTcBImg), &full[s]);
          issued |= 1u << s;
          parity = (parity & ~(1u << s)) | ((r & 1) << s);
        }
      }
      // after an abort: let copies still in flight land before the CTA exits
      if (*abort_flag) {
        for (int s = 0; s < kTcStages; ++s) {
          if (!((issued >> s) & 1)) continue;
          const long long t0 = clock64();
          while (!mbar_try(&full[s], (parity >> s) & 1) && clock64() - t0 < kWaitCycles) {
          }
        }
      }
    }
    __syncwarp();
  } else if (warp == 1) {
    // ------------------------------------------------------------ MMA issuer
    // (one thread: its chain of waits and MMAs must stay shorter than the
    // epilogue's work on a half tile)
    if (elect_one()) {
    uint32_t g = 0, v = 0, u[kTcPair] = {};
    const uint64_t da0 = mat_desc(su32(aimg), 128, 512), dx0 = mat_desc(su32(xs), 128, 512);
    constexpr uint32_t kK16 = 256 >> 4;  // descriptor steps (16 bytes): 16 columns on,
    constexpr uint32_t kALo = uint32_t(kTcAImg) >> 4, kXLo = uint32_t(kTcBImg) >> 4;  // hi image to lo image
    for (int64_t pt = pt0; pt < pt1; pt += kTcPair, ++v) {
      const int ab = int(v & 1);
      const int tiles = pt + 1 < pt1 ? 2 : 1;
      const bool have_a = mbar_wait(&afull[ab], (v >> 1) & 1, abort_flag);
      const uint64_t dab = da0 + uint64_t(2 * kTcPair * ab * kALo);
      for (int j = 0; j < 2 * nx; ++j, ++g) {
        const int s = int(g % kTcStages);
        const bool have_x = have_a && mbar_wait(&full[s], (g / kTcStages) & 1, abort_flag);
        const uint64_t dx = dx0 + uint64_t(uint32_t(s) * (uint32_t(kTcStageBytes) >> 4));
#pragma unroll
        for (int t = 0; t < kTcPair; ++t) {
          if (t >= tiles) break;
          const uint32_t b = u[t] & 1, ph = (u[t] >> 1) & 1;
          ++u[t];
          if (!have_x || !mbar_wait(&tempty[2 * t + b], ph ^ 1, abort_flag)) continue;
          tc_fence_after();
          {
            const uint32_t dcol = tmem + (2 * t + b) * uint32_t(kTcRows);
            const uint64_t da = dab + uint64_t(2 * t * kALo);
            mma_bf16<0>(dcol, da, dx);
            mma_bf16<1>(dcol, da + kALo, dx);
            mma_bf16<1>(dcol, da, dx + kXLo);
            mma_bf16<1>(dcol, da + kK16, dx + kK16);
            mma_bf16<1>(dcol, da + kALo + kK16, dx + kK16);
            mma_bf16<1>(dcol, da + kK16, dx + kXLo + kK16);
            mma_commit(&tfull[2 * t + b]);
          }
        }
        if (have_x) mma_commit(&empty[s]);
      }
      // the A images of this pass are free once its MMAs have completed
      if (have_a) mma_commit(&aempty[ab]);
    }
    }
    __syncwarp();
  } else if (warp < 4) {
    // ------------------------------------------------------------ A image stager
    const int ts = threadIdx.x - 64;
    uint32_t v = 0;
    for (int64_t pass = pt0; pass < pt1; pass += kTcPair, ++v) {
      const int ab = int(v & 1);
      const int tiles = pass + 1 < pt1 ? 2 : 1;
      const bool free_buf = mbar_wait_warp(&aempty[ab], ((v >> 1) & 1) ^ 1, abort_flag);
      for (int tl = 0; free_buf && tl < tiles; ++tl) {
        const int64_t pt = pass + tl;
        const int t = ts;
        uint8_t* ahi = aimg + size_t(2 * (kTcPair * ab + tl)) * kTcAImg;
        uint8_t* alo = ahi + kTcAImg;
        // every load of the thread is issued before the conversions, so the
        // tile's memory latency is paid about once (with few data tiles per
        // particle tile -- small M -- this staging sets the kernel's pace)
        if ((d & 3) == 0) {
          // 16-byte loads: thread t takes the groups e = t + 64 u of four
          // consecutive features (r = e / 8, k = 4 (e % 8)); a row of d
          // features is d / 4 such groups, the rest of the 32 are zero
          constexpr int kG = kTcPT * kLgK / 4 / kTcStageThreads;  // 16
          float4 vals[kG];
#pragma unroll
          for (int u = 0; u < kG; ++u) {
            const int e = t + kTcStageThreads * u;
            const int r = e >> 3, k = (e & 7) << 2;
            const int64_t i = pt * kTcPT + r;
            vals[u] = (i < n && k < d) ? *reinterpret_cast<const float4*>(x + i * d + k)
                                       : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
          }
#pragma unroll
          for (int u = 0; u < kG; ++u) {
            const int e = t + kTcStageThreads * u;
            const int r = e >> 3, k = (e & 7) << 2;
            const float f[4] = {vals[u].x, vals[u].y, vals[u].z, vals[u].w};
            uint16_t hi[4], lo[4];
#pragma unroll
            for (int c = 0; c < 4; ++c) {
              hi[c] = bf16_rn(f[c]);
              lo[c] = bf16_rn(f[c] - __uint_as_float(uint32_t(hi[c]) << 16));
            }
            // features k .. k + 3 are adjacent in the core-matrix image
            *reinterpret_cast<uint2*>(ahi + img_off(r, k)) =
                make_uint2(uint32_t(hi[0]) | (uint32_t(hi[1]) << 16), uint32_t(hi[2]) | (uint32_t(hi[3]) << 16));
            *reinterpret_cast<uint2*>(alo + img_off(r, k)) =
                make_uint2(uint32_t(lo[0]) | (uint32_t(lo[1]) << 16), uint32_t(lo[2]) | (uint32_t(lo[3]) << 16));
          }
        } else {
          constexpr int kB = 8;  // loads in flight per thread
          for (int e0 = t; e0 < kTcPT * kLgK; e0 += kTcStageThreads * kB) {
            float vals[kB];
#pragma unroll
            for (int u = 0; u < kB; ++u) {
              const int e = e0 + kTcStageThreads * u;
              const int r = e / kLgK, k = e % kLgK;
              const int64_t i = pt * kTcPT + r;
              vals[u] = (i < n && k < d) ? x[i * d + k] : 0.0f;
            }
#pragma unroll
            for (int u = 0; u < kB; ++u) {
              const int e = e0 + kTcStageThreads * u;
              const int r = e / kLgK, k = e % kLgK;
              const uint16_t hi = bf16_rn(vals[u]);
              const uint16_t lo = bf16_rn(vals[u] - __uint_as_float(uint32_t(hi) << 16));
              *reinterpret_cast<uint16_t*>(ahi + img_off(r, k)) = hi;
              *reinterpret_cast<uint16_t*>(alo + img_off(r, k)) = lo;
            }
          }
        }
      }
      if (free_buf) asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      mbar_arrive(&afull[ab]);
      // the FP64 part of log pi for each particle (two per thread and tile),
      // kept off the epilogue warps: b.(v - w / 2) - |b|^2 / (2 prior_var).
      // Slot v % 4 is free: writing pass v requires the MMAs of pass v - 2 to
      // have completed, hence the epilogue to have finished pass v - 4.
      if (!*abort_flag) {
        double* pre = s_pre + size_t(v % kTcPreRing) * kTcPair * kTcPT;
        for (int r = ts; r < tiles * kTcPT; r += kTcStageThreads) {
          const int64_t i = pass * kTcPT + r;
          double bv = 0.0, b2 = 0.0;
          if (i < n) {
            const float* xi = x + i * d;
#pragma unroll 4
            for (int c = 0; c < d; ++c) {
              const double bc = widen(xi[c]);
              bv = fma(bc, tg->vw[c], bv);
              b2 = fma(bc, bc, b2);
            }
          }
          pre[r] = bv - b2 / (2.0 * tg->prior_var);
        }
      }
      mbar_arrive(&prefull[v % kTcPreRing]);
    }
  } else {
    // ------------------------------------------------------------ epilogue
    // particle tile tl of the pass; column group 2 p + hh of each image tile
    // (64 of its 256 rows) comes with half tile p
    const int q = warp & 3, grp = (warp - 4) >> 2, tl = grp >> 1, hh = grp & 1;
    const int row = 32 * q + lane;
    uint32_t v = 0, u = 0;
    const double log2_pad = double(tg->m_pad - tg->m);
    for (int64_t pass = pt0; pass < pt1; pass += kTcPair, ++v) {
      if (pass + tl >= pt1) break;  // (only the last pass can lack its second tile)
      const int64_t i = (pass + tl) * kTcPT + row;
      // what the pass's end needs, loaded before its work
      double lw0 = 0.0;
      float lp0 = 0.0f;
      if (hh == 0 && i < n) {
        lw0 = a.logw[i];
        lp0 = lp[i];
      }
      // sums over up to 8 image tiles, and their totals as FP32 pairs
      float fabs4[2] = {0.0f, 0.0f}, flg4[2] = {0.0f, 0.0f};
      float sa[2] = {0.0f, 0.0f}, sal[2] = {0.0f, 0.0f}, sg[2] = {0.0f, 0.0f}, sgl[2] = {0.0f, 0.0f};
      // A warp always has the load of its next 32 columns in flight, across
      // half tiles too, while it processes the 32 before them: the wait for
      // the MMAs, the load's latency and the hand-over of the buffer are
      // hidden behind the exponentials.  The buffer goes back to the MMA warp
      // as soon as its last columns have arrived.
      uint32_t z[2][16];
      const uint32_t tq = tmem + (uint32_t(32 * q) << 16) + uint32_t(2 * tl * kTcRows + hh * 64);
      // |z| log2 e (the images are scaled): the sum and the running product
      // in column order
      auto process = [&](const uint32_t (&zz)[16], float& fa, float& fl) {
        float prod = 1.0f;
#pragma unroll
        for (int e = 0; e < 16; ++e) {
          const float az = fabsf(__uint_as_float(zz[e]));
          fa += az;
          prod = fmaf(prod, ex2_approx(-az), prod);
        }
        fl += lg2_approx(prod);
      };
      // (the waits' outcomes are warp-uniform: tcgen05.ld is a warp-collective;
      // after a failed one the numbers do not matter, the tile is not written)
      bool ok = mbar_wait_warp(&tfull[2 * tl], (u >> 1) & 1, abort_flag);
      tc_fence_after();
      if (ok) tmem_ld16(tq, z[0]);
      for (int j = 0; j < nx; ++j) {
#pragma unroll
        for (int p = 0; p < 2; ++p, ++u) {
#pragma unroll
          for (int c = 0; c < 4; ++c) {
            tmem_wait_ld(z[c & 1]);
            if (c < 3) {
              if (ok) tmem_ld16(tq + uint32_t(p * kTcRows + 16 * (c + 1)), z[(c + 1) & 1]);
            } else {
              tc_fence_before();
              __syncwarp();
              if (lane == 0) mbar_arrive(&tempty[2 * tl + p]);
              if (p == 0 || j + 1 < nx) {
                ok = mbar_wait_warp(&tfull[2 * tl + (p ^ 1)], ((u + 1) >> 1) & 1, abort_flag);
                tc_fence_after();
                if (ok) tmem_ld16(tq + uint32_t((p ^ 1) * kTcRows), z[0]);
              }
            }
            process(z[c & 1], fabs4[p], flg4[p]);
          }
        }
        if ((j & 7) == 7 || j == nx - 1) {
#pragma unroll
          for (int p = 0; p < 2; ++p) {
            add_pair(fabs4[p] * kAbsScale, sa[p], sal[p]);
            add_pair(flg4[p], sg[p], sgl[p]);
            fabs4[p] = flg4[p] = 0.0f;
          }
        }
      }
      double acc_abs[2], acc_lg[2];
#pragma unroll
      for (int p = 0; p < 2; ++p) {
        acc_abs[p] = pair_value(sa[p], sal[p]) * (1.0 / double(kAbsScale));
        acc_lg[p] = pair_value(sg[p], sgl[p]);
      }
      double* sp = s_part + (tl * kTcPT + row) * 4;
      if (hh == 1) {
#pragma unroll
        for (int p = 0; p < 2; ++p) {
          sp[2 * p] = acc_abs[p];
          sp[2 * p + 1] = acc_lg[p];
        }
      }
      named_sync(2 + tl, kTcTileThreads);
      if (hh == 0) {
        // the constant term of this tile (written by the stager warps)
        const bool have_pre = mbar_wait_warp(&prefull[v % kTcPreRing], (v / kTcPreRing) & 1, abort_flag);
        if (i < n && have_pre && !*abort_flag) {
          const double sum_abs = ((acc_abs[0] + sp[0]) + acc_abs[1]) + sp[2];
          const double sum_lg = (((acc_lg[0] - log2_pad) + sp[1]) + acc_lg[1]) + sp[3];
          const double ln2 = 0.6931471805599453;
          const float lpn = float(s_pre[((v % kTcPreRing) * kTcPair + tl) * kTcPT + row] - 0.5 * ln2 * sum_abs - ln2 * sum_lg);
          // eq. (5): the log-target difference in FP32 (exact when the two
          // values are within a factor of two), one FP64 addition
          const double lw = lw0 + double(lpn - lp0);
          lp[i] = lpn;
          a.logw[i] = lw;
          mt.add(lw);
        }
      }
      named_sync(2 + tl, kTcTileThreads);  // partial sums read before the next pass writes them
    }
  }

  // ------------------------------------------------------------ block maximum, teardown
  __syncwarp();
  {
    const long long wm = warp_max_ll(mt.best);
    const int wn = __any_sync(0xffffffffu, mt.nan);
    if (lane == 0) {
      wmax[warp] = wm;
      wnan[warp] = wn;
    }
  }
  tc_fence_before();
  __syncthreads();
  if (threadIdx.x == 0) {
    long long v = wmax[0];
    int nan = wnan[0];
    for (int w = 1; w < kTcWarps; ++w) {
      v = wmax[w] > v ? wmax[w] : v;
      nan |= wnan[w];
    }
    if (a.flags & PA_FUSED_ITER) {
      atomicMax(&a.st->mkey, v);
    } else {
      a.part[2 * blockIdx.x] = from_ordered_key(v);
      a.part[2 * blockIdx.x + 1] = 1.0;
    }
    if (nan) record_error(a.st, SMC_ENONFINITE);
    if (*abort_flag) record_error(a.st, SMC_ETIMEOUT);
  }
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTcCols) : "memory");
  }
}

}  // namespace

int logistic_tc_grid(int64_t n, int sms) {
  const int64_t npt = (n + kTcPT - 1) / kTcPT;
  return int(npt < sms ? npt : sms);
}

cudaError_t launch_logistic_tc(const ParticleArgs& a, int grid, cudaStream_t s) {
  // the dynamic shared-memory limit is a per-device attribute of the kernel
  static std::atomic<bool> configured[64];
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
  if (!configured[dev].load()) {
    e = cudaFuncSetAttribute(k_logistic_tc, cudaFuncAttributeMaxDynamicSharedMemorySize, int(kTcSmem));
    if (e != cudaSuccess) return e;
    configured[dev].store(true);
  }
  chain_launch(k_logistic_tc, grid, kTcThreads, kTcSmem, s, a);
  return cudaGetLastError();
}

}  // namespace smc
