// FP64-accurate dense products on the BF16 tensor cores, by exact 8-bit digits (Ozaki's error-free splitting).
//
// Why: the Gram matrices and block updates of the solvers are n x q x q products.  GB300's FP64 tensor path runs at
// 1.1 TFLOP/s, tcgen05 at 1,900 in BF16.  Every operand entry becomes seven signed 8-bit digits (55 bits below the
// largest entry of its row or column); BF16 holds a digit, and FP32 a sum of 1,024 digit products, exactly.  The 28
// products of digits i + j <= 6 are summed exactly, the six of i + j = 7 in FP32, so an entry C_pq is off by at most
//   2^-56 (e_p |b_q|_1 + e_q |a_p|_1) + K 2^-61 e_p e_q,   e: the power of two above the largest entry,
// from the digits below the 55th bit and the products of i + j >= 8.  Measured against exact sums, unit columns:
// normal entries 2e-16 (the FP64 tensor path 8e-16); columns localised on one of 300,000 rows 5.4e-15 on the diagonal
// (1.3e-15 to 4e-15; at 3,000 rows 2e-16 and 2e-15), as the squares of a column's fifth digits all add up, and 6e-17 off
// it.  With i + j <= 6 alone (28 products) those were 1.6e-14 and 1e-14; the 34 take 1.2 times as long (300,000 x 994:
// Gram 13.5 -> 16.3 ms, update 26.6 -> 32.5; on the FP64 tensor path 341 and 563).
// All this is relative to the columns' largest entries: an entry of C that sums small products only (columns whose
// large entries lie in different rows) keeps fewer digits than in FP64.
//
// Sums.  The digit products of equal weight i + j = g share one TMEM accumulator (128 x 64 FP32, eight of them: all
// 512 columns).  After 128 terms (7 x 128 x 2^14 < 2^24) the epilogue warps add them as integers into two 64-bit sums
// a tile element, hi (g = 0..3) and lo (g = 4..7), value hi 2^32 + lo.  The last weight, g = 7, needs no exact sum (its
// rounding in FP32 is 2^-23 of 2^-53): it stays in its accumulator until the tile ends.  The integers of the tile's
// split are added by atomics, the same bits in any order.  lo grows by up to 2^40.4 a term: K <= 2^22 at once
// (kDigitTerms).
//
// Layout.  The digits lie in memory as the tensor cores' K-major core matrices (8 rows x 16 bytes), ordered
// [block of 32 k][digit][8 rows][4 x 8 k], so a tile's operand is seven contiguous pieces a stage, fetched by bulk
// copies into the order that the descriptors name.  Two stages of 32 k (86 KB each).
//
// Roles: warp 0 copies, warp 1 issues the MMAs, warps 2 to 9 drain (two a TMEM lane quarter, 32 columns each).
// A group's accumulator is free for the next 128 terms as soon as it is drained, so the MMAs wait for the first
// group only.  Every wait has a limit; a CTA that gives up sets *err, and the result becomes NaN.
#include <cmath>

#include "pfe_internal.h"

namespace pfe {
namespace {

constexpr int kDigits = 7;
constexpr int kTM = 128, kTN = 64, kBK = 32;  // tile and stage
constexpr int kChunk = 4;                     // stages between two drains: 128 terms
constexpr int kPieceA = kTM * kBK * 2, kPieceB = kTN * kBK * 2;
constexpr int kStageBytes = kDigits * (kPieceA + kPieceB);
constexpr int kSmem = 2 * kStageBytes + 256;
constexpr int kThreads = 320;
constexpr int32_t kNoExp = -100000;   // exponent of a row or column of zeros
constexpr int32_t kNotFinite = 100000;  // ... with an Inf or NaN

__device__ __forceinline__ uint32_t smem_of(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void bar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void bar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void bar_expect(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ uint64_t now_ns() {
  uint64_t t;
  asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
  return t;
}
// true when the phase completed, false after two seconds
__device__ __forceinline__ bool bar_wait(uint32_t bar, uint32_t parity) {
  uint64_t t0 = 0;
  for (uint32_t i = 0;; ++i) {
    uint32_t ok;
    asm volatile(
        "{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\nselp.u32 %0, 1, 0, p;\n}"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    if (ok) return true;
    if ((i & 63) == 63) {
      const uint64_t t = now_ns();
      if (t0 == 0) t0 = t;
      else if (t - t0 > 2000000000ull) return false;
    }
  }
}
__device__ __forceinline__ void bulk_copy(uint32_t dst, const void *src, uint32_t bytes, uint32_t bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
               "l"(src), "r"(bytes), "r"(bar)
               : "memory");
}
// K-major operand without swizzle: 128 bytes between core matrices along k, 512 between groups of eight rows
__device__ __forceinline__ uint64_t operand(uint32_t addr) {
  return (uint64_t)((addr >> 4) & 0x3fff) | ((uint64_t)(128 >> 4) << 16) | ((uint64_t)(512 >> 4) << 32) |
         ((uint64_t)1 << 46);
}
constexpr uint32_t kInstr = (1u << 4) | (1u << 7) | (1u << 10) | ((kTN >> 3) << 17) | ((kTM >> 4) << 24);  // F32 += BF16 BF16
__device__ __forceinline__ void mma(uint32_t d, uint64_t a, uint64_t b, uint32_t accumulate) {
  asm volatile(
      "{\n.reg .pred p;\nsetp.ne.u32 p, %4, 0;\ntcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}" ::"r"(d),
      "l"(a), "l"(b), "r"(kInstr), "r"(accumulate)
      : "memory");
}
__device__ __forceinline__ void mma_commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar)
               : "memory");
}
__device__ __forceinline__ void fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
// 32 columns of this warp's TMEM lanes
__device__ __forceinline__ void tmem_load(uint32_t addr, uint32_t (&v)[32]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,%19,"
      "%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];\n"
      "tcgen05.wait::ld.sync.aligned;"
      : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]), "=r"(v[8]),
        "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15]), "=r"(v[16]),
        "=r"(v[17]), "=r"(v[18]), "=r"(v[19]), "=r"(v[20]), "=r"(v[21]), "=r"(v[22]), "=r"(v[23]), "=r"(v[24]),
        "=r"(v[25]), "=r"(v[26]), "=r"(v[27]), "=r"(v[28]), "=r"(v[29]), "=r"(v[30]), "=r"(v[31])
      : "r"(addr)
      : "memory");
}
// a b + c in one instruction (see fixed_step.cu)
__device__ __forceinline__ int64_t mad(int32_t a, int32_t b, int64_t c) {
  int64_t d;
  asm("mul.wide.s32 %0, %1, %2;" : "=l"(d) : "r"(a), "r"(b));
  return d + c;
}

// (hi 2^32 + lo) 2^e rounded to double, by integer operations (the FP64 pipe would take as long as the MMAs)
__device__ double to_double(int64_t hi, int64_t lo, int32_t e) {
  hi += lo >> 32;
  uint32_t l = (uint32_t)lo;
  const bool neg = hi < 0;
  if (neg) {  // negate the 96-bit value
    hi = ~hi + (l == 0 ? 1 : 0);
    l = 0u - l;
  }
  if (hi == 0 && l == 0) return 0.0;
  const int z = hi ? __clzll(hi) : 64 + __clz((int)l) - 0;
  // 64 leading bits m of the value, m 2^(e + 32 - z) (hi == 0: shift the low word up)
  uint64_t m;
  bool sticky = false;
  if (hi) {
    m = z == 0 ? (uint64_t)hi : ((uint64_t)hi << z) | (z >= 32 ? (uint64_t)l << (z - 32) : (uint64_t)(l >> (32 - z)));
    if (z < 32) sticky = z == 0 ? l != 0 : (l << z) != 0;
  } else {
    m = (uint64_t)l << (z - 64 + 32);
  }
  int32_t x = e + 32 - z + 63;  // exponent of the leading bit
  uint64_t q = m >> 11;
  const uint32_t rest = (uint32_t)m & 0x7ff;
  if (rest > 0x400 || (rest == 0x400 && (sticky || (q & 1)))) ++q;
  if (q >> 53) {
    q >>= 1;
    ++x;
  }
  const double mag = x > 1023 ? __longlong_as_double(0x7ff0000000000000ll)
                     : x < -1022 ? ldexp((double)q, x - 52)
                                 : __longlong_as_double((long long)((q & 0xfffffffffffffull) | ((uint64_t)(x + 1023) << 52)));
  return neg ? -mag : mag;
}

// One tile of the product of two digit operands over stages [kb0, kb1), as (hi, lo) per thread: row `lane of the
// tile` x 32 columns, in the epilogue warps.  Returns false in threads whose role gave up.
struct Tile {
  const uint16_t *A, *B;  // digits
  int64_t ga, gb;         // groups of eight rows of the operands
  int64_t ra, rb;         // first group of this tile
  int32_t kb0, kb1;
};

__device__ __forceinline__ bool tile_product(const Tile &t, unsigned char *smem, int64_t (&hi)[32], int64_t (&lo)[32]) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t bars = smem_of(smem + 2 * kStageBytes);
  const uint32_t full = bars, empty = bars + 16, done = bars + 32, free_g = bars + 40;  // 2, 2, 1, 7 barriers
  uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(smem + 2 * kStageBytes + 128);
  if (threadIdx.x == 0) {
    for (int s = 0; s < 2; ++s) {
      bar_init(full + 8 * s, 1);
      bar_init(empty + 8 * s, 1);
    }
    bar_init(done, 1);
    for (int g = 0; g < kDigits; ++g) bar_init(free_g + 8 * g, 8);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(smem_of(tmem_slot)) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  fence_before();
  __syncthreads();
  fence_after();
  const uint32_t tmem = *tmem_slot;
  const int32_t stages = t.kb1 - t.kb0;
  bool ok = true;
  if (warp == 0) {
    if (lane == 0) {
      int32_t it = 0;
      for (; it < stages; ++it) {
        const int s = it & 1;
        if (it >= 2 && !bar_wait(empty + 8 * s, ((it >> 1) - 1) & 1)) {
          ok = false;
          break;
        }
        bar_expect(full + 8 * s, kStageBytes);
        const uint32_t dst = smem_of(smem + s * kStageBytes);
        for (int d = 0; d < kDigits; ++d) {
          const int64_t slice = (int64_t)(t.kb0 + it) * kDigits + d;
          bulk_copy(dst + d * kPieceA, t.A + (slice * t.ga + t.ra) * 256, kPieceA, full + 8 * s);
          bulk_copy(dst + kDigits * kPieceA + d * kPieceB, t.B + (slice * t.gb + t.rb) * 256, kPieceB, full + 8 * s);
        }
      }
      // the copies in flight have landed before the CTA ends
      for (int32_t b = max(0, it - 2); b < it; ++b) bar_wait(full + 8 * (b & 1), (b >> 1) & 1);
    }
  } else if (warp == 1) {
    if (lane == 0) {
      for (int32_t it = 0; it < stages && ok; ++it) {
        const int s = it & 1;
        ok = bar_wait(full + 8 * s, (it >> 1) & 1);
        if (!ok) break;
        fence_after();
        const int32_t chunk = it / kChunk;
        const bool first = it % kChunk == 0;
        const uint32_t a0 = smem_of(smem + s * kStageBytes), b0 = a0 + kDigits * kPieceA;
        const auto pair = [&](int g, int i, bool fresh) {
          for (int kk = 0; kk < kBK / 16; ++kk)
            mma(tmem + g * kTN, operand(a0 + i * kPieceA + kk * 256), operand(b0 + (g - i) * kPieceB + kk * 256),
                !(fresh && kk == 0));
        };
        for (int g = 0; g < kDigits && ok; ++g) {
          if (first && chunk > 0) {
            ok = bar_wait(free_g + 8 * g, (chunk - 1) & 1);
            if (!ok) break;
            fence_after();
          }
          for (int i = 0; i <= g; ++i) pair(g, i, first && i == 0);
        }
        if (!ok) break;
        for (int i = 1; i < kDigits; ++i) pair(kDigits, i, it == 0 && i == 1);
        mma_commit(empty + 8 * s);
        if (it % kChunk == kChunk - 1 || it == stages - 1) mma_commit(done);
      }
    }
  } else {
    const int quarter = warp & 3, half = (warp - 2) >> 2;
    const uint32_t base = tmem + ((uint32_t)(32 * quarter) << 16) + 32 * half;
    const int32_t chunks = (stages + kChunk - 1) / kChunk;
    for (int32_t c = 0; c < chunks; ++c) {
      ok = __all_sync(0xffffffffu, bar_wait(done, c & 1));  // the TMEM loads are the whole warp's
      if (!ok) break;
      fence_after();
#pragma unroll
      for (int g = 0; g < kDigits; ++g) {
        uint32_t v[32];
        tmem_load(base + g * kTN, v);
        fence_before();
        __syncwarp();
        if (lane == 0) bar_arrive(free_g + 8 * g);
#pragma unroll
        for (int e = 0; e < 32; ++e) {
          const int32_t n = __float2int_rn(__uint_as_float(v[e]));
          if (g < 4) hi[e] = mad(n, 1 << (8 * (3 - g)), hi[e]);
          else lo[e] = mad(n, 1 << (8 * (7 - g)), lo[e]);
        }
      }
    }
    if (ok) {  // the last weight
      uint32_t v[32];
      tmem_load(base + kDigits * kTN, v);
#pragma unroll
      for (int e = 0; e < 32; ++e) lo[e] += __float2ll_rn(__uint_as_float(v[e]));
    }
  }
  __syncwarp();
  return ok;
}

__device__ __forceinline__ void tile_end(unsigned char *smem) {
  uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(smem + 2 * kStageBytes + 128);
  fence_before();
  __syncthreads();
  fence_after();
  if ((threadIdx.x >> 5) == 1)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(*tmem_slot) : "memory");
}

// Gram tiles: hi, lo sums added to acc (column-major mp x np, hi then lo); the stages split over blockIdx.z.
// sym: tiles that lie below the diagonal are left to the mirrored ones.
__global__ void __launch_bounds__(kThreads, 1) k_gram_digits(const uint16_t *A, const uint16_t *B, int32_t mp, int32_t np,
                                                             int32_t stages, int32_t per_split, int sym,
                                                             unsigned long long *acc, int32_t *err) {
  extern __shared__ __align__(1024) unsigned char smem[];
  if (sym && ((int)blockIdx.y + 1) * kTN <= (int)blockIdx.x * kTM) return;
  Tile t{A, B, mp / 8, np / 8, (int64_t)blockIdx.x * (kTM / 8), (int64_t)blockIdx.y * (kTN / 8),
         (int32_t)blockIdx.z * per_split, min(stages, ((int32_t)blockIdx.z + 1) * per_split)};
  if (t.kb0 >= t.kb1) return;
  int64_t hi[32], lo[32];
#pragma unroll
  for (int e = 0; e < 32; ++e) hi[e] = lo[e] = 0;
  if (!tile_product(t, smem, hi, lo)) *err = 1;
  const int warp = threadIdx.x >> 5;
  if (warp >= 2) {
    const int64_t p = (int64_t)blockIdx.x * kTM + 32 * (warp & 3) + (threadIdx.x & 31);
    const int64_t q0 = (int64_t)blockIdx.y * kTN + 32 * ((warp - 2) >> 2);
#pragma unroll
    for (int e = 0; e < 32; ++e) {
      unsigned long long *c = acc + (q0 + e) * mp + p;
      atomicAdd(c, (unsigned long long)hi[e]);
      atomicAdd(c + (int64_t)mp * np, (unsigned long long)lo[e]);
    }
  }
  tile_end(smem);
}

// C[q ldc + p] = alpha 2^(..) (hi 2^32 + lo) + beta C; with sym the tiles left out are mirrored
__global__ void k_gram_finish(int32_t m, int32_t nn, int32_t mp, int32_t np, const long long *__restrict__ acc,
                              const int32_t *__restrict__ ea, const int32_t *__restrict__ eb, double alpha, double beta,
                              double *C, int64_t ldc, int sym, const int32_t *err) {
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= (int64_t)m * nn) return;
  const int32_t q = (int32_t)(t / m), p = (int32_t)(t - (int64_t)q * m);
  const bool mirror = sym && (q / kTN + 1) * kTN <= p / kTM * kTM;
  const int32_t sp = mirror ? q : p, sq = mirror ? p : q;
  const int64_t at = (int64_t)sq * mp + sp;
  const int32_t a = ea[sp], b = eb[sq];
  double v = to_double(acc[at], acc[at + (int64_t)mp * np], a == kNoExp || b == kNoExp ? 0 : a + b - 110 + 40);
  if (a == kNotFinite || b == kNotFinite || *err) v = __longlong_as_double(0x7ff8000000000000ll);
  C[(int64_t)q * ldc + p] = alpha * v + (beta == 0.0 ? 0.0 : beta * C[(int64_t)q * ldc + p]);
}

// C (rows x N row-major) = alpha A B + beta C over all stages; upper: column tile [q0, q0 + 64) needs k < q0 + 64
__global__ void __launch_bounds__(kThreads, 1) k_update_digits(const uint16_t *A, const uint16_t *B, int64_t rows, int64_t rp,
                                                               int32_t N, int32_t np, int32_t stages, int upper,
                                                               const int32_t *__restrict__ ea,
                                                               const int32_t *__restrict__ eb, double alpha, double beta,
                                                               double *C, int64_t ldc) {
  extern __shared__ __align__(1024) unsigned char smem[];
  const int32_t last = upper ? min(stages, ((int32_t)blockIdx.x + 1) * kTN / kBK) : stages;
  Tile t{A, B, rp / 8, np / 8, (int64_t)blockIdx.y * (kTM / 8), (int64_t)blockIdx.x * (kTN / 8), 0, last};
  int64_t hi[32], lo[32];
#pragma unroll
  for (int e = 0; e < 32; ++e) hi[e] = lo[e] = 0;
  const bool ok = tile_product(t, smem, hi, lo);
  const int failed = __syncthreads_or(!ok);
  const int warp = threadIdx.x >> 5;
  if (warp >= 2) {
    const int64_t i = (int64_t)blockIdx.y * kTM + 32 * (warp & 3) + (threadIdx.x & 31);
    const int32_t q0 = (int32_t)blockIdx.x * kTN + 32 * ((warp - 2) >> 2);
    if (i < rows) {
      const int32_t a = ea[i];
      double *c = C + i * ldc + q0;
#pragma unroll
      for (int e = 0; e < 32; ++e) {
        if (q0 + e >= N) break;
        const int32_t b = __ldg(eb + q0 + e);
        double v = to_double(hi[e], lo[e], a == kNoExp || b == kNoExp ? 0 : a + b - 110 + 40);
        if (failed || a == kNotFinite || b == kNotFinite) v = __longlong_as_double(0x7ff8000000000000ll);
        c[e] = alpha * v + (beta == 0.0 ? 0.0 : beta * c[e]);
      }
    }
  }
  tile_end(smem);
}

// ---- exponents and digits ---------------------------------------------------------------------
// e with |x| < 2^e; zero: kNoExp, Inf and NaN: kNotFinite (a denormal counts as 2^-1022)
__device__ __forceinline__ int32_t exponent_of(uint64_t bits) {
  const int32_t x = (int32_t)(bits >> 52) & 0x7ff;
  if (x == 0x7ff) return kNotFinite;
  if (x == 0) return (bits << 1) ? -1021 : kNoExp;
  return x - 1022;
}
// x 2^(55 - e) rounded to nearest
__device__ __forceinline__ int64_t fixed_of(uint64_t bits, int32_t e) {
  const int32_t x = (int32_t)(bits >> 52) & 0x7ff;
  if (x == 0x7ff) return 0;
  uint64_t m = bits & 0xfffffffffffffull;
  if (x) m |= 1ull << 52;
  const int32_t sh = (x ? x : 1) - 1075 + 55 - e;
  const int64_t v = sh >= 0 ? (int64_t)(m << min(sh, 10)) : sh < -60 ? 0 : (int64_t)((m + (1ull << (-sh - 1))) >> -sh);
  return (int64_t)bits < 0 ? -v : v;
}
// the seven digits of eight values, as pairs of BF16: out[d] holds digit d of v[0..7]
__device__ __forceinline__ void digits_of(int64_t (&v)[8], uint4 (&out)[kDigits]) {
#pragma unroll
  for (int d = kDigits - 1; d >= 0; --d) {
    uint32_t w[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const int32_t n = d ? (int32_t)(int8_t)(uint8_t)v[k] : (int32_t)v[k];
      v[k] = (v[k] - n) >> 8;
      w[k] = __float_as_uint((float)n);
    }
    out[d] = make_uint4(__byte_perm(w[0], w[1], 0x7632), __byte_perm(w[2], w[3], 0x7632), __byte_perm(w[4], w[5], 0x7632),
                        __byte_perm(w[6], w[7], 0x7632));
  }
}

// largest exponent of each column of a row-major block into e (set to kNoExp before); finite_only leaves Inf and NaN out
__global__ void __launch_bounds__(256) k_col_exponent(int64_t K, int32_t m, const uint64_t *__restrict__ X, int64_t ld,
                                                      int64_t slab, int finite_only, int32_t *e) {
  __shared__ int32_t red[8][33];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int32_t c = blockIdx.y * 32 + lane;
  const int64_t r0 = (int64_t)blockIdx.x * slab, r1 = min(K, r0 + slab);
  int32_t x = kNoExp;
  if (c < m)
    for (int64_t i = r0 + warp; i < r1; i += 8) {
      const int32_t t = exponent_of(X[i * ld + c]);
      x = finite_only && t == kNotFinite ? x : max(x, t);
    }
  red[warp][lane] = x;
  __syncthreads();
  if (warp == 0 && c < m) {
    for (int w = 1; w < 8; ++w) x = max(x, red[w][lane]);
    if (x > kNoExp) atomicMax(e + c, x);
  }
}
__global__ void k_set_exponents(int32_t *e, int64_t n) {
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t < n) e[t] = kNoExp;
}

// Digits of rows [r0, r0 + 32 stages) of a row-major block, contraction along the rows: operand rows are the columns
__global__ void __launch_bounds__(256) k_digits_cols(int64_t r0, int64_t K, int32_t m, int32_t mp,
                                                     const uint64_t *__restrict__ X, int64_t ld,
                                                     const int32_t *__restrict__ e, uint16_t *out) {
  const int32_t c = blockIdx.y * 64 + (threadIdx.x & 63), kg = threadIdx.x >> 6;
  const int64_t row = r0 + (int64_t)blockIdx.x * kBK + kg * 8;
  int64_t v[8];
  const int32_t ec = c < m ? e[c] : kNoExp;
#pragma unroll
  for (int k = 0; k < 8; ++k)
    v[k] = (c < m && row + k < K && ec > kNoExp && ec < kNotFinite) ? fixed_of(X[(row + k) * ld + c], ec) : 0;
  uint4 w[kDigits];
  digits_of(v, w);
#pragma unroll
  for (int d = 0; d < kDigits; ++d)
    reinterpret_cast<uint4 *>(out)[((((int64_t)blockIdx.x * kDigits + d) * (mp / 8) + c / 8) * 4 + kg) * 8 + (c & 7)] = w[d];
}

// Digits of rows whose K entries lie along memory, entry k times 2^(sign ek[k]): one CTA per eight rows, their
// exponents into e
__global__ void __launch_bounds__(256) k_digits_rows(int64_t rows, int64_t rp, int32_t K, int32_t stages,
                                                     const uint64_t *__restrict__ X, int64_t ld,
                                                     const int32_t *__restrict__ ek, int sign, int32_t *e, uint16_t *out) {
  __shared__ int32_t red[32][8];
  const int r8 = threadIdx.x & 7, col = threadIdx.x >> 3;  // 32 groups of eight k
  const int64_t row = (int64_t)blockIdx.x * 8 + r8;
  const uint64_t *x = X + row * ld;
  int32_t er = kNoExp;
  if (row < rows)
    for (int32_t k = col; k < K; k += 32) {
      const int32_t t = exponent_of(x[k]), s = ek[k];
      if (t == kNotFinite) er = kNotFinite;
      else if (t > kNoExp && er < kNotFinite) er = max(er, s > kNoExp ? t + sign * s : t);
    }
  red[col][r8] = er;
  __syncthreads();
  for (int w = 16; w > 0; w >>= 1) {
    if (col < w) red[col][r8] = max(red[col][r8], red[col + w][r8]);
    __syncthreads();
  }
  er = red[0][r8];
  if (col == 0 && row < rp) e[row] = er;
  for (int32_t kg = col; kg < stages * 4; kg += 32) {
    int64_t v[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const int32_t c = kg * 8 + k;
      v[k] = 0;
      if (row < rows && c < K && er > kNoExp && er < kNotFinite) {
        const int32_t s = ek[c];
        v[k] = fixed_of(x[c], s > kNoExp ? er - sign * s : er);
      }
    }
    uint4 w[kDigits];
    digits_of(v, w);
#pragma unroll
    for (int d = 0; d < kDigits; ++d)
      reinterpret_cast<uint4 *>(out)[((((int64_t)(kg >> 2) * kDigits + d) * (rp / 8) + blockIdx.x) * 4 + (kg & 3)) * 8 + r8] = w[d];
  }
}

int64_t up(int64_t x, int64_t a) { return (x + a - 1) / a * a; }
// Digits of one operand held at a time: written and read again within L2 (129 MB), and little beside a solve's blocks
constexpr int64_t kSlabBytes = 64ll << 20;

// rows of a slab whose digits take at most kSlabBytes (a multiple of 128)
int64_t slab_rows(int64_t rows, int64_t width) {
  return std::min(up(rows, 128), std::max<int64_t>(128, kSlabBytes / (2 * kDigits * width) / 128 * 128));
}

void column_exponents(int64_t K, int32_t m, const double *X, int64_t ld, bool finite_only, int32_t *e, int64_t len,
                      cudaStream_t s) {
  PFE_LAUNCH k_set_exponents<<<(unsigned)((len + 255) / 256), 256, 0, s>>>(e, len);
  const int64_t parts = std::max<int64_t>(1, std::min<int64_t>((K + 255) / 256, 256)), slab = (K + parts - 1) / parts;
  PFE_LAUNCH k_col_exponent<<<dim3((unsigned)parts, (unsigned)((m + 31) / 32)), 256, 0, s>>>(
      K, m, reinterpret_cast<const uint64_t *>(X), ld, slab, finite_only ? 1 : 0, e);
}

template <typename F>
void allow_smem(F *kernel) {
  cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmem);
}

}  // namespace

// workspace: err (64 bytes), exponents, the sums, the digits of both operands
size_t digit_gram_bytes(int64_t K, int32_t m, int32_t nn, bool same) {
  const int64_t mp = up(m, kTM), np = up(nn, kTM);
  const int64_t rows = slab_rows(K, std::max(mp, np));
  return 64 + 4 * (mp + np) + 16 * mp * np + 2 * kDigits * rows * (mp + (same ? 0 : np)) + 1024;
}

void launch_gram_digits(int64_t K, int32_t m, int32_t nn, const double *A, int64_t lda, const double *B, int64_t ldb,
                        double alpha, double beta, double *C, int64_t ldc, bool sym, void *work, cudaStream_t s) {
  const bool same = A == B && lda == ldb && m == nn;
  const int32_t mp = (int32_t)up(m, kTM), np = (int32_t)up(nn, kTM);
  const int64_t rows = slab_rows(K, std::max(mp, np));
  char *w = static_cast<char *>(work);
  int32_t *err = reinterpret_cast<int32_t *>(w), *ea = err + 16, *eb = same ? ea : ea + mp;
  w += 64 + 4 * ((int64_t)mp + np);
  w = reinterpret_cast<char *>(up((int64_t)reinterpret_cast<uintptr_t>(w), 256));
  unsigned long long *acc = reinterpret_cast<unsigned long long *>(w);
  w += 16 * (int64_t)mp * np;
  uint16_t *da = reinterpret_cast<uint16_t *>(w), *db = same ? da : da + (int64_t)kDigits * rows * mp;
  cudaMemsetAsync(err, 0, 64, s);
  cudaMemsetAsync(acc, 0, 16 * (size_t)mp * np, s);
  column_exponents(K, m, A, lda, false, ea, mp, s);
  if (!same) column_exponents(K, nn, B, ldb, false, eb, np, s);
  allow_smem(k_gram_digits);
  const int tp = (m + kTM - 1) / kTM, tq = (nn + kTN - 1) / kTN;
  int tiles = 0;
  for (int p = 0; p < tp; ++p)
    for (int q = 0; q < tq; ++q) tiles += !(sym && (q + 1) * kTN <= p * kTM);
  for (int64_t r0 = 0; r0 < K; r0 += rows) {
    const int32_t stages = (int32_t)(up(std::min(rows, K - r0), 32 * kChunk) / kBK);
    PFE_LAUNCH k_digits_cols<<<dim3(stages, mp / 64), 256, 0, s>>>(r0, K, m, mp, reinterpret_cast<const uint64_t *>(A), lda,
                                                                   ea, da);
    if (!same)
      PFE_LAUNCH k_digits_cols<<<dim3(stages, np / 64), 256, 0, s>>>(r0, K, nn, np, reinterpret_cast<const uint64_t *>(B),
                                                                     ldb, eb, db);
    // one CTA an SM: as many splits as fill the GPU once, whole chunks each
    const int32_t chunks = stages / kChunk;
    const int32_t want = std::max(1, std::min(chunks, 152 / std::max(tiles, 1)));
    const int32_t per = (chunks + want - 1) / want * kChunk;
    PFE_LAUNCH k_gram_digits<<<dim3(tp, tq, (stages + per - 1) / per), kThreads, kSmem, s>>>(da, db, mp, np, stages, per,
                                                                                             sym ? 1 : 0, acc, err);
  }
  const int64_t tot = (int64_t)m * nn;
  PFE_LAUNCH k_gram_finish<<<(unsigned)((tot + 255) / 256), 256, 0, s>>>(
      m, nn, mp, np, reinterpret_cast<const long long *>(acc), ea, eb, alpha, beta, C, ldc, sym ? 1 : 0, err);
}

size_t digit_update_bytes(int64_t M, int32_t N, int32_t K) {
  const int64_t kp = up(K, 128), np = up(N, kTM), rows = slab_rows(M, kp);
  return 4 * (kp + np + rows) + 2 * kDigits * kp * (rows + np) + 1024;
}

void launch_update_digits(int64_t M, int32_t N, int32_t K, const double *A, int64_t lda, const double *Bc, int64_t ldb,
                          double alpha, double beta, double *C, int64_t ldc, bool upper, void *work, cudaStream_t s) {
  const int32_t kp = (int32_t)up(K, 128), np = (int32_t)up(N, kTM), stages = kp / kBK;
  const int64_t rows = slab_rows(M, kp);
  int32_t *ek = static_cast<int32_t *>(work), *eb = ek + kp, *ea = eb + np;
  char *w = reinterpret_cast<char *>(up((int64_t)reinterpret_cast<uintptr_t>(ea + rows), 256));
  uint16_t *db = reinterpret_cast<uint16_t *>(w), *da = db + (int64_t)kDigits * kp * np;
  // Columns of A are brought to one magnitude by powers of two that go to the rows of B: an entry then only meets
  // digits of its own scale (the filtered block's columns differ in norm, and R^-1 undoes it)
  column_exponents(M, K, A, lda, true, ek, kp, s);
  PFE_LAUNCH k_digits_rows<<<(unsigned)(np / 8), 256, 0, s>>>(N, np, K, stages, reinterpret_cast<const uint64_t *>(Bc), ldb,
                                                              ek, 1, eb, db);
  allow_smem(k_update_digits);
  for (int64_t r0 = 0; r0 < M; r0 += rows) {
    const int64_t cnt = std::min(rows, M - r0), rp = up(cnt, kTM);
    PFE_LAUNCH k_digits_rows<<<(unsigned)(rp / 8), 256, 0, s>>>(
        cnt, rp, K, stages, reinterpret_cast<const uint64_t *>(A + r0 * lda), lda, ek, -1, ea, da);
    PFE_LAUNCH k_update_digits<<<dim3((unsigned)((N + kTN - 1) / kTN), (unsigned)(rp / kTM)), kThreads, kSmem, s>>>(
        da, db, cnt, rp, N, np, stages, upper ? 1 : 0, ea, eb, alpha, beta, C + r0 * ldc, ldc);
  }
}

}  // namespace pfe
