// The FP64 filter (Alg. 2) in 64-bit fixed point.
//
// Why: GB300 issues 2 FP64 FMAs a clock and SM, but about 30 32 x 32 + 64-bit multiply-adds (IMAD.WIDE, measured)
// and 64 to 128 of the simpler integer operations.  A multiply-add of two 60-bit numbers is three IMAD.WIDE, a
// fifth of the time of one FP64 FMA, and the step leaves the FP64 pipe, where it ran at 0.9 of its rate.
//
// Numbers.  A Chebyshev vector is stored as (h, l) pairs of int32: value (h 2^30 + l) 2^-sh with l in
// [-2^29, 2^29) and one exponent sh per column and vector; |h| <= 2^30.  The operator A = (2/d)(H - cI) is stored
// in the same split, U = u 2^60 = uh 2^30 + ul (full blocks: a 2^59).  A product keeps
//   uh xh 2^60 + (uh xl + ul xh) 2^30     (two 64-bit sums, accH and accM; ul xl 2^-60 <= 2^-2 of a unit is dropped)
// and a sum over a row is rounded once, (accH + (accM + 2^29) >> 30), in units of the input vector.  A column's
// largest entry times ||A||_inf + 1 fills 60 bits, so for ||A||_inf near 6 a typical entry has 55 bits, and a step
// adds about half a unit of rounding to it, 2^-56: the FMA chain of a row takes 13 to 40 roundings of 2^-53.
// Measured against 128-bit arithmetic with the same operator (relative 2-norm of a column): 0.9e-15 (FP64 kernels
// 1.6e-15) at degree 40, 1.9e-15 (2.6e-15) at 301, 0.3e-15 (1.4e-15) with full blocks.  Errors are relative to a
// column's largest entry, as the recurrence mixes the entries of a column.
//
// Scaling.  Each step knows, per column, bounds M on the |h| of t_j and t_{j-1} and the exponents, so every CTA
// derives the same shift o of the new vector from
//   |t_{j+1}| <= ||A||_inf |t_j| + |t_{j-1}|  <  2^60:
// right when that could overflow, left when two or more bits would lie idle.  In a filter whose spectrum lies
// in [-1, 1] the shift is almost always 0; vectors that grow (a bound below the spectrum) or spread (a start
// concentrated on few atoms) move their exponent.  M of the new vector is an atomic maximum that starts at 1/16
// of a recent one, so that few lanes write.  State: 4 rotating slots of sh and M per column.
//
// Columns with an Inf, a NaN or a largest entry beyond 2^+-800 keep doubles in the same buffers and take the FP64 FMAs
// inside the same kernel (kRaw), so every input gives what it gave before.  With the largest coefficient between
// 2^-100 and 2^60 one unit of the result, 2^-60 of the column's largest term, is then a normal double.
#include <algorithm>
#include <cmath>

#include "pfe_internal.h"

namespace pfe {
namespace {

constexpr int kLimb = 30;                    // bits of the low limb
constexpr int32_t kMask = (1 << kLimb) - 1;  // low limb of a non-negative remainder
constexpr int32_t kHalf = 1 << (kLimb - 1);
constexpr int32_t kRaw = INT32_MIN;          // exponent of a column kept in FP64

// The full product.  As assembly with the addition outside it becomes one multiply-add; the C product of two
// loaded words becomes three multiplies, and mad.wide a multiply and a separate addition (2.8 x, 1.5 x the
// instructions of a block).
__device__ __forceinline__ int64_t mul(int32_t a, int32_t b) {
  int64_t d;
  asm("mul.wide.s32 %0, %1, %2;" : "=l"(d) : "r"(a), "r"(b));
  return d;
}
__device__ __forceinline__ int64_t mad(int32_t a, int32_t b, int64_t c) { return mul(a, b) + c; }

// (h, l) of a 64-bit value: h rounded to nearest, l the signed rest
__device__ __forceinline__ int2 split(int64_t v) {
  const int64_t t = v + kHalf;
  return make_int2((int32_t)((uint32_t)t & kMask) - kHalf, (int32_t)(t >> kLimb));
}
__device__ __forceinline__ int64_t join(int2 p) { return mad(p.y, 1 << kLimb, (int64_t)p.x); }
// v 2^o, rounded to nearest for o < 0
__device__ __forceinline__ int64_t shifted(int64_t v, int o) {
  if (o >= 0) return o > 62 ? 0 : (int64_t)((uint64_t)v << o);
  return o < -62 ? 0 : (v + ((int64_t)1 << (-o - 1))) >> -o;
}
// Exact up to one rounding to double; two FP64 additions (the conversion instruction runs at 2 a clock as well).  The
// two halves take the exponents 2^52 and 2^84, a known method (compiler-rt's __floatundidf).
__device__ __forceinline__ double to_double(int64_t v) {
  const uint32_t lo = (uint32_t)v, hi = (uint32_t)((uint64_t)v >> 32) ^ 0x80000000u;
  const double dl = __hiloint2double(0x43300000, (int)lo);  // 2^52 + lo
  const double dh = __hiloint2double(0x45300000, (int)hi);  // 2^84 + (hi + 2^31) 2^32
  return (dh - 0x1.00000801p84) + dl;                      // 2^84 + 2^63 + 2^52
}
__device__ __forceinline__ double pow2(int e) {
  return __hiloint2double(e < -1022 ? 0 : (min(e, 1024) + 1023) << 20, 0);  // 0 and Inf outside the range
}

// the exponent clipped to [-126, 90]
__device__ __forceinline__ float pow2f(int e) { return __int_as_float((min(max(e, -126), 90) + 127) << 23); }

// Plain loads: under programmatic launch the buffers are still being written when this grid's CTAs start, so the
// read-only path, whose data may not change during a grid's life, is not open to them.
template <int CPL>
__device__ __forceinline__ void load_pairs(const int2 *p, int2 (&v)[CPL]) {
  if constexpr (CPL == 2) {
    const int4 t = *reinterpret_cast<const int4 *>(p);
    v[0] = make_int2(t.x, t.y);
    v[1] = make_int2(t.z, t.w);
  } else {
    v[0] = *p;
  }
}
template <int CPL>
__device__ __forceinline__ void store_pairs(int2 *p, const int2 (&v)[CPL]) {
  if constexpr (CPL == 2)
    *reinterpret_cast<int4 *>(p) = make_int4(v[0].x, v[0].y, v[1].x, v[1].y);
  else
    *p = v[0];
}
template <int CPL>
__device__ __forceinline__ void load_y(const double *p, double (&v)[CPL]) {
  if constexpr (CPL == 2) {
    const double2 t = *reinterpret_cast<const double2 *>(p);
    v[0] = t.x;
    v[1] = t.y;
  } else {
    v[0] = *p;
  }
}
template <int CPL>
__device__ __forceinline__ void store_y(double *p, const double (&v)[CPL]) {
  if constexpr (CPL == 2)
    *reinterpret_cast<double2 *>(p) = make_double2(v[0], v[1]);
  else
    *p = v[0];
}
template <int CPL>
__device__ __forceinline__ void load_state(const int32_t *p, int32_t (&v)[CPL]) {
  if constexpr (CPL == 2) {
    const int2 t = *reinterpret_cast<const int2 *>(p);
    v[0] = t.x;
    v[1] = t.y;
  } else {
    v[0] = *p;
  }
}

// arguments of one step (j -> j + 1)
struct StepArgs {
  int32_t n_atoms;
  int32_t groups, tile;      // CPL-wide column groups per row; of them per CTA
  int32_t per_pass, passes;  // atoms of a CTA at a time, and how often
  uint32_t magic;            // division of a lane's slot by tile: (slot magic) >> 16
  int64_t ld;
  const int32_t *rp;     // row starts: off-diagonal blocks (rank-1) or all blocks (full)
  const int4 *blk;       // rank-1: two int4 per block (u0, u1 | u2, column, 0); full: five (nine pairs, column, 0)
  const int4 *dg;        // rank-1: six pairs per atom (three int4), negated
  const double *u64, *d64;  // the same operator in FP64 for the columns kept in FP64
  const int32_t *ci64;
  const int32_t *info;   // see note_row
  const int2 *X, *W;
  int2 *Z;
  double *Y;
  int32_t *sh, *mx;      // [4][kc]
  int64_t kc;
  int32_t j;
  int2 ga, gb;           // g_j, g_{j+1} times 2^(kLimb * 2 - 1 - ge), split
  int32_t ge;
  double g0, g1;         // the same coefficients
  // MODE_EMIT, MODE_ADJ: Y receives the new vector in FP64, times 2^emit
  int32_t emit;
  // MODE_ADJ: Z = A X (halved: / 2) - W + g0 Ybar, Ybar in fixed point with its exponents and bounds
  const int2 *Ybar;
  const int32_t *ybar_sh, *ybar_mx;
  int32_t halved;
};
constexpr int MODE_EMIT = 5;  // as MODE_STEP, Y = Z

// The FP64 form of the step for one lane's columns (an input with Inf, NaN or extreme magnitudes).
template <int CPL, int MODE, bool FULL>
__device__ __noinline__ void raw_step(const StepArgs &a, int64_t atom, int64_t c0) {
  const double *X = reinterpret_cast<const double *>(a.X);
  const double *W = reinterpret_cast<const double *>(a.W);
  double *Z = reinterpret_cast<double *>(a.Z);
  for (int c = 0; c < CPL; ++c) {
    double acc[3] = {0.0, 0.0, 0.0};
    const double *xo = X + 3 * atom * a.ld + c0 + c;
    if (!FULL) {
      const double *d = a.d64 + 6 * atom;
      const double x0 = xo[0], x1 = xo[a.ld], x2 = xo[2 * a.ld];
      acc[0] = fma(d[0], x0, fma(d[1], x1, d[2] * x2));
      acc[1] = fma(d[1], x0, fma(d[3], x1, d[4] * x2));
      acc[2] = fma(d[2], x0, fma(d[4], x1, d[5] * x2));
    }
    for (int p = a.rp[atom]; p < a.rp[atom + 1]; ++p) {
      const int64_t col = a.ci64[p];
      const double *x = X + 3 * col * a.ld + c0 + c;
      const double x0 = x[0], x1 = x[a.ld], x2 = x[2 * a.ld];
      if (FULL) {
        const double *v = a.u64 + 9 * (int64_t)p;
        for (int r = 0; r < 3; ++r) acc[r] = fma(v[3 * r], x0, fma(v[3 * r + 1], x1, fma(v[3 * r + 2], x2, acc[r])));
      } else {
        const double *u = a.u64 + 3 * (int64_t)p;
        const double s = fma(u[0], x0, fma(u[1], x1, u[2] * x2));
        for (int r = 0; r < 3; ++r) acc[r] = fma(-s, u[r], acc[r]);
      }
    }
    for (int r = 0; r < 3; ++r) {
      const int64_t off = (3 * atom + r) * a.ld + c0 + c;
      double z = MODE == MODE_FIRST ? 0.5 * acc[r] : (MODE == MODE_ADJ && a.halved ? 0.5 : 1.0) * acc[r] - W[off];
      if (MODE == MODE_ADJ) z = fma(a.g0, reinterpret_cast<const double *>(a.Ybar)[off], z);
      Z[off] = z;
      if (MODE == MODE_EMIT || MODE == MODE_ADJ) a.Y[off] = ldexp(z, a.emit);
      else if (MODE == MODE_FIRST) a.Y[off] = fma(a.g1, z, a.g0 * X[off]);
      else if (MODE == MODE_STEP_ACC) a.Y[off] = fma(a.g0, X[off], fma(a.g1, z, a.Y[off]));
      else if (a.Y) a.Y[off] = fma(a.g1, z, a.Y[off]);
    }
  }
}

// What the operator allows: the bits of a stored value (64 hold (||A||_inf + 1) of them) and the blocks whose
// cross terms 64 bits hold.
__device__ __forceinline__ float norm_of(const int32_t *info) { return fmaxf(__int_as_float(__ldg(info + 1)), 2.f); }
__device__ __forceinline__ int top_of(const int32_t *info, float g) {
  const int by_norm = g < 6.9f ? 60 : g < 14.9f ? 59 : 58;
  // the high limb of u . x takes |u|_1 2^(top - 30) < 2^31
  return __int_as_float(__ldg(info + 5)) < 1.9f ? by_norm : min(by_norm, 59);
}
// rank-1 blocks between two folds (two always fit, see k_fixed_r1)
__device__ __forceinline__ int fold_of(const int32_t *info) {
  return __int_as_float(__ldg(info + 2)) < 15.5f ? 6 : __int_as_float(__ldg(info + 3)) < 15.5f ? 4 : 2;
}

template <int CPL>
__device__ __forceinline__ void load_atom(const char *xl, uint32_t col, uint32_t stride, int64_t ldb, int2 (&x)[3][CPL]) {
  const char *p = xl + (uint64_t)col * stride;
  load_pairs<CPL>(reinterpret_cast<const int2 *>(p), x[0]);
  load_pairs<CPL>(reinterpret_cast<const int2 *>(p + ldb), x[1]);
  load_pairs<CPL>(reinterpret_cast<const int2 *>(p + 2 * ldb), x[2]);
}

// accH, accM += (3 x 3 block v) x, v nine pairs
template <int CPL>
__device__ __forceinline__ void add_block(const int2 (&v)[9], const int2 (&x)[3][CPL], int64_t (&accH)[3][CPL],
                                          int64_t (&accM)[3][CPL]) {
#pragma unroll
  for (int r = 0; r < 3; ++r)
#pragma unroll
    for (int s = 0; s < 3; ++s)
#pragma unroll
      for (int c = 0; c < CPL; ++c) {
        accH[r][c] = mad(v[3 * r + s].y, x[s][c].y, accH[r][c]);
        accM[r][c] = mad(v[3 * r + s].y, x[s][c].x, accM[r][c]);
        accM[r][c] = mad(v[3 * r + s].x, x[s][c].y, accM[r][c]);
      }
}

// accH, accM += u (u . x); start: half a unit for the rounding of u . x, plus half a limb so that its low limb comes
// out signed.  A register: as a constant it costs two additions a column (62 instructions a block instead of 56).
template <int CPL>
__device__ __forceinline__ void add_rank1(int64_t start, const int4 &b0, const int4 &b1, const int2 (&x)[3][CPL],
                                          int64_t (&accH)[3][CPL], int64_t (&accM)[3][CPL]) {
  const int2 u[3] = {make_int2(b0.x, b0.y), make_int2(b0.z, b0.w), make_int2(b1.x, b1.y)};
#pragma unroll
  for (int c = 0; c < CPL; ++c) {
    int64_t H = mul(u[0].y, x[0][c].y), M = mad(u[0].y, x[0][c].x, start);
    M = mad(u[0].x, x[0][c].y, M);
#pragma unroll
    for (int r = 1; r < 3; ++r) {
      H = mad(u[r].y, x[r][c].y, H);
      M = mad(u[r].y, x[r][c].x, M);
      M = mad(u[r].x, x[r][c].y, M);
    }
    const int64_t t = H + (M >> kLimb);
    const int32_t sl = (int32_t)((uint32_t)t & kMask) - kHalf, s = (int32_t)(t >> kLimb);
#pragma unroll
    for (int r = 0; r < 3; ++r) {
      accH[r][c] = mad(u[r].y, s, accH[r][c]);
      accM[r][c] = mad(u[r].y, sl, accM[r][c]);
      accM[r][c] = mad(u[r].x, s, accM[r][c]);
    }
  }
}

template <int CPL, bool FULL>
__device__ __forceinline__ void add_neighbour(int64_t start, const int4 *w, const int2 (&x)[3][CPL], int64_t (&accH)[3][CPL],
                                              int64_t (&accM)[3][CPL]) {
  if (FULL) {
    int2 v[9];
#pragma unroll
    for (int t = 0; t < 4; ++t) {
      v[2 * t] = make_int2(w[t].x, w[t].y);
      v[2 * t + 1] = make_int2(w[t].z, w[t].w);
    }
    v[8] = make_int2(w[4].x, w[4].y);
    add_block<CPL>(v, x, accH, accM);
  } else {
    add_rank1<CPL>(start, w[0], w[1], x, accH, accM);
  }
}

template <int CPL>
__device__ __forceinline__ void fold(int64_t (&accH)[3][CPL], int64_t (&accM)[3][CPL]) {
#pragma unroll
  for (int r = 0; r < 3; ++r)
#pragma unroll
    for (int c = 0; c < CPL; ++c) {
      accH[r][c] += accM[r][c] >> kLimb;
      accM[r][c] &= kMask;
    }
}

// What a lane needs to know of a column besides its entries
struct ColumnScale {
  int32_t o, wsh;  // shift of the new vector; exponent of t_j minus that of t_{j-1}
  double ysc;      // value of one unit of the filter sum's increment
};

// One fused step.  A CTA owns `tile` column groups (CPL columns each) and per_pass atoms at a time, a lane one
// atom and one group; its atoms' blocks (contiguous in the block list) and its columns' scales sit in shared
// memory, so the neighbour loop's only global loads are the gathers, and passes > 1 spreads the set-up over
// several atoms.
// What bounds it: the gathers' latency at 24 warps an SM, and the pipe of the multiplies.  IMAD.WIDE runs at about 30 a
// clock and SM (measured), 18 a block and column make 165 us of the step at N = 99,900, k = 64; its pipe is 52 to 57 %
// busy (ncu, N = 29,600, k = 64), with most stalls on the gathers.  A step moves 614 MB at N = 99,900, 91 us at 6.76
// TB/s (ncu: DRAM 22 %, L2 20 % busy).  Measured against the FP64 kernels: 876 -> 280 us a step (k = 64), 13.8 -> 4.37 ms
// (k = 994), full blocks 250 -> 81 us (N = 20,000, k = 64).
// 24 warps an SM (80 registers).  Rank-1: CTAs of 128 lanes and one gather at a time; a second gather in flight
// spills (303 us with 80 registers, 309 with 96), as do 64 registers (296).  Full blocks have three times the
// products a gather and gain from it (81 against 89 us).  Prefetching rows to L1 or L2 only added instructions
// (309, 340 us), as did four lanes an atom where the GPU is not full (N = 1,000, k = 16: 8.9 us either way).
template <int CPL, int MODE, bool FULL>
__global__ void __launch_bounds__(256, 3) k_fixed_step(const StepArgs a) {
  constexpr int kWords = FULL ? 5 : 2;  // int4 per block
  extern __shared__ int4 smem[];
  ColumnScale *scale = reinterpret_cast<ColumnScale *>(smem);
  int4 *sblk = smem + a.tile * CPL;
  const uint32_t slot = threadIdx.x, mine = (slot * a.magic) >> 16;
  const int32_t group = blockIdx.y * a.tile + (int32_t)(slot - mine * a.tile);
  const int32_t c0 = group * CPL;
  const int32_t first = blockIdx.x * (a.per_pass * a.passes), last = min(first + a.per_pass * a.passes, a.n_atoms);
  const int sj = a.j & 3, sp = (a.j + 3) & 3, sn = (a.j + 1) & 3, sr = (a.j + 2) & 3;
  // ---- the blocks of this CTA's atoms, then the scales of its columns.  The operator is complete before a filter's
  // first step, so the next step's CTAs may start, and stage their blocks, while this one's last CTAs run.
  asm volatile("griddepcontrol.launch_dependents;");
  const int32_t pbase = __ldg(a.rp + first);
  {
    const int32_t words = (__ldg(a.rp + last) - pbase) * kWords;
    const int4 *src = a.blk + (int64_t)pbase * kWords;
    for (int32_t t = threadIdx.x; t < words; t += blockDim.x) sblk[t] = __ldg(src + t);
  }
  asm volatile("griddepcontrol.wait;" ::: "memory");  // the previous step is complete and visible
  for (int32_t t = threadIdx.x; t < a.tile * CPL; t += blockDim.x) {
    const int64_t c = (int64_t)blockIdx.y * a.tile * CPL + t;
    if (c >= a.kc) break;
    const int32_t mj = a.mx[sj * a.kc + c], shj = a.sh[sj * a.kc + c];
    const float g = norm_of(a.info);  // >= 2: t_j itself also fits the new scale
    ColumnScale q{};
    float bound = g * (float)(mj + 1);
    bool zero = mj == 0;
    if (MODE == MODE_FIRST || (MODE == MODE_ADJ && a.halved)) bound *= 0.5f;
    if (MODE != MODE_FIRST) {
      const int32_t mp = a.mx[sp * a.kc + c];
      q.wsh = shj - a.sh[sp * a.kc + c];
      bound += (float)(mp + 1) * pow2f(q.wsh);
      zero = zero && mp == 0;
    }
    // g_j Ybar can exceed a_{j+1} by any factor (g_m far below the other coefficients): its exponent `term` stays an
    // integer, and the sum is bounded in units of 2^far where it passes the range of float
    int far = 0;
    if (MODE == MODE_ADJ) {
      const int32_t my = a.ybar_mx[c];
      if (my != 0 && a.ga.y != 0) {
        const int term = a.ge + (shj - a.ybar_sh[c]);
        far = max(0, term - 60);
        bound = bound * pow2f(-far) + (float)(abs(a.ga.y) + 1) * 0x1p-29f * (float)(my + 1) * pow2f(term - far);
      }
      zero = zero && my == 0;
    }
    // bound 1.001 < 2^e: room for top - kLimb - e more bits
    const int e = ((__float_as_int(bound * 1.001f) >> 23) & 255) - 126 + far;
    const int room = top_of(a.info, g) - kLimb - e;
    q.o = zero ? 0 : room < 0 ? room : room > 1 ? room - 1 : 0;
    q.ysc = pow2((MODE == MODE_EMIT || MODE == MODE_ADJ ? a.emit : a.ge + 1) - (shj + q.o));
    scale[t] = q;
    if (blockIdx.x == 0) {
      a.sh[sn * a.kc + c] = shj == kRaw ? kRaw : shj + q.o;
      a.mx[sr * a.kc + c] = mj >> 4;  // start of the next vector's maximum
    }
  }
  __syncthreads();
  if ((int32_t)mine >= a.per_pass || group >= a.groups) return;
  const bool raw = a.sh[sj * a.kc + c0] == kRaw;
  const ColumnScale *sc = scale + (slot - mine * a.tile) * CPL;
  bool plain = true;
  int32_t big[CPL];
#pragma unroll
  for (int c = 0; c < CPL; ++c) {
    plain = plain && sc[c].o == 0 && (MODE == MODE_FIRST || sc[c].wsh == 0);
    big[c] = 0;
  }
  int64_t start = (int64_t)kHalf + ((int64_t)kHalf << kLimb);
  asm volatile("" : "+l"(start));
  const int64_t ldb = a.ld * 8;
  const uint32_t stride = (uint32_t)(3 * ldb);
  const char *xl = reinterpret_cast<const char *>(a.X + c0);
  const bool with_y = MODE != MODE_STEP || a.Y != nullptr;
  int32_t ysh[CPL];
  if (MODE == MODE_ADJ && !raw)
    for (int c = 0; c < CPL; ++c) ysh[c] = a.sh[sj * a.kc + c0 + c] - a.ybar_sh[c0 + c] + a.ge + 1;
  for (int32_t atom = first + (int32_t)mine; atom < last; atom += a.per_pass) {
    if (raw) {
      raw_step<CPL, MODE, FULL>(a, atom, c0);
      continue;
    }
    int64_t accH[3][CPL], accM[3][CPL];
#pragma unroll
    for (int r = 0; r < 3; ++r)
#pragma unroll
      for (int c = 0; c < CPL; ++c) {
        accH[r][c] = 0;
        accM[r][c] = FULL ? kHalf / 2 : kHalf;  // the final rounding
      }
    int32_t p = __ldg(a.rp + atom) - pbase;
    const int32_t p1 = __ldg(a.rp + atom + 1) - pbase;
    int2 x0[3][CPL];
    const auto load = [&](int32_t q, int2 (&x)[3][CPL]) {
      load_atom<CPL>(xl, (uint32_t)sblk[q * kWords + kWords - 1].z, stride, ldb, x);
    };
    if (FULL) {
      // the gather of the next block is in flight during the products of one; two blocks between folds
      int2 x1[3][CPL];
      if (p < p1) load(p, x0);
      for (; p + 1 < p1; p += 2) {
        load(p + 1, x1);
        add_neighbour<CPL, FULL>(start, sblk + p * kWords, x0, accH, accM);
        if (p + 2 < p1) load(p + 2, x0);
        add_neighbour<CPL, FULL>(start, sblk + (p + 1) * kWords, x1, accH, accM);
        fold<CPL>(accH, accM);
      }
      if (p < p1) add_neighbour<CPL, FULL>(start, sblk + p * kWords, x0, accH, accM);
    } else {
      load_atom<CPL>(xl, (uint32_t)atom, stride, ldb, x0);
      const int4 d0 = __ldg(a.dg + 3 * (int64_t)atom), d1 = __ldg(a.dg + 3 * (int64_t)atom + 1),
                 d2 = __ldg(a.dg + 3 * (int64_t)atom + 2);
      const int2 xx = make_int2(d0.x, d0.y), xy = make_int2(d0.z, d0.w), xz = make_int2(d1.x, d1.y),
                 yy = make_int2(d1.z, d1.w), yz = make_int2(d2.x, d2.y), zz = make_int2(d2.z, d2.w);
      const int2 v[9] = {xx, xy, xz, xy, yy, yz, xz, yz, zz};
      add_block<CPL>(v, x0, accH, accM);
      const int32_t kFold = fold_of(a.info);
      int32_t until = kFold;
      for (; p < p1; ++p) {
        load(p, x0);
        add_neighbour<CPL, FULL>(start, sblk + p * kWords, x0, accH, accM);
        if (--until == 0) {
          fold<CPL>(accH, accM);
          until = kFold;
        }
      }
    }
#pragma unroll
    for (int r = 0; r < 3; ++r) {
      const int64_t off = (3 * (int64_t)atom + r) * a.ld + c0;
      int2 z[CPL], w[CPL], xo[CPL];
      double y[CPL];
      constexpr bool kEmit = MODE == MODE_EMIT || MODE == MODE_ADJ;
      if (MODE != MODE_FIRST) load_pairs<CPL>(a.W + off, w);
      if (MODE == MODE_FIRST || MODE == MODE_STEP_ACC) load_pairs<CPL>(a.X + off, xo);
      if (MODE == MODE_ADJ) load_pairs<CPL>(a.Ybar + off, xo);
      if (MODE != MODE_FIRST && !kEmit && with_y) load_y<CPL>(a.Y + off, y);
#pragma unroll
      for (int c = 0; c < CPL; ++c) {
        int64_t v = FULL ? (accH[r][c] << 1) + (accM[r][c] >> (kLimb - 1)) : accH[r][c] + (accM[r][c] >> kLimb);
        if (MODE == MODE_FIRST) {
          v = shifted(-v, sc[c].o - 1);
        } else if (MODE == MODE_ADJ) {
          const int64_t P = mad(a.ga.y, xo[c].y, mad(a.ga.x, xo[c].y, mad(a.ga.y, xo[c].x, kHalf)) >> kLimb);
          // each term at the new scale: at the old one g Ybar could exceed 64 bits beside a small a_{j+1}
          v = shifted(-v, sc[c].o - a.halved) - shifted(join(w[c]), sc[c].wsh + sc[c].o) + shifted(P, ysh[c] + sc[c].o);
        } else if (plain) {
          v = -v - join(w[c]);
        } else {
          v = shifted(-v - shifted(join(w[c]), sc[c].wsh), sc[c].o);
        }
        z[c] = split(v);
        big[c] = max(big[c], abs(z[c].y));
        if (kEmit) y[c] = to_double(v) * sc[c].ysc;
      }
      store_pairs<CPL>(a.Z + off, z);
      if (kEmit) {
        store_y<CPL>(a.Y + off, y);
      } else if (with_y) {
#pragma unroll
        for (int c = 0; c < CPL; ++c) {
          int64_t H = mad(a.gb.y, z[c].y, 0), M = mad(a.gb.x, z[c].y, mad(a.gb.y, z[c].x, kHalf));
          if (MODE == MODE_FIRST || MODE == MODE_STEP_ACC) {
            if (!plain) xo[c] = split(shifted(join(xo[c]), sc[c].o));
            H = mad(a.ga.y, xo[c].y, H);
            M = mad(a.ga.x, xo[c].y, mad(a.ga.y, xo[c].x, M));
          }
          const double t = to_double(H + (M >> kLimb));
          y[c] = MODE == MODE_FIRST ? t * sc[c].ysc : fma(t, sc[c].ysc, y[c]);
        }
        store_y<CPL>(a.Y + off, y);
      }
    }
  }
  if (raw) return;
#pragma unroll
  for (int c = 0; c < CPL; ++c) {
    int32_t *m = a.mx + sn * a.kc + c0 + c;
    if (big[c] > *reinterpret_cast<volatile int32_t *>(m)) atomicMax(m, big[c]);
  }
}

// ---- the operator in fixed point -------------------------------------------------------------
__device__ __forceinline__ int2 fixed_entry(double v, double unit) {
  const int64_t t = __double2ll_rn(v * unit);
  // +2 in units of 2^-60 (an atom without neighbours): one limb down from 2^31
  return t > ((int64_t)1 << 61) - kHalf - 1 ? make_int2((int32_t)(t - ((int64_t)INT32_MAX << kLimb)), INT32_MAX) : split(t);
}

// *p = max(*p, v) for non-negative values, with an atomic only where it would change
__device__ __forceinline__ void raise(int32_t *p, int32_t v) {
  if (v > *reinterpret_cast<volatile int32_t *>(p)) atomicMax(p, v);
}
// info[0] |= 1 when the operator does not fit; info[1]: ||A||_inf as float bits, rounded up
__device__ __forceinline__ void note_row(int32_t *info, double row, bool bad) {
  if (bad || !(row <= 16.0)) atomicOr(info, 1);
  else raise(info + 1, __float_as_int(__double2float_ru(row * 1.000001)));
}
// sums and maxima over the 16 lanes of an atom
__device__ __forceinline__ double sum16(double v) {
  for (int d = 8; d > 0; d >>= 1) v += __shfl_xor_sync(0xffffffffu, v, d);
  return v;
}
__device__ __forceinline__ float max16(float v) {
  for (int d = 8; d > 0; d >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, d));
  return v;
}
__device__ __forceinline__ bool any16(bool v) {
  return (__ballot_sync(0xffffffffu, v) >> (threadIdx.x & 16) & 0xffffu) != 0;
}

// Both kernels take 16 lanes an atom: with one a row's chain of FP64 conversions took 42 us at N = 800, as long as six
// filter steps (10 us now), and a first call of few steps was slower than in the FP64 kernels.
//
// Rank-1 form, unit 2^-60.  With |x| < 2^60 the cross terms of a row's diagonal block and F of its other blocks
// stay below 2^59 (3 + sum |d| + sum (|u_r| + |u|_1)), which 63 bits hold for a factor below 15.5: info[2], info[3]
// get the largest one for F = 6, 4.  An operator whose factor for F = 2 is larger does not fit, nor does one with
// |u|_1 >= 3.9 (the high limb of u . x would leave 32 bits, see top_of).  Neither occurs while the bound holds
// (||A||_2 <= 2: |u|_2 <= sqrt(2), a diagonal row below 3.5).  info[4]: the longest row, info[5]: the largest |u|_1.
// The factors are sums of floats, a relative 1e-5 up.  A pass takes 12 blocks, two groups of six, three of four.
__global__ void __launch_bounds__(128) k_fixed_r1(int32_t n_atoms, const int32_t *__restrict__ rp1,
                                                  const int32_t *__restrict__ ci1, const double *__restrict__ u,
                                                  const double *__restrict__ dg, int4 *blk, int2 *dgo, int32_t *info) {
  const int64_t i = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 4;
  const int lane = threadIdx.x & 15;
  const bool live = i < n_atoms;
  double row[3] = {0.0, 0.0, 0.0};
  float drow = 0.f;
  bool bad = false;
  if (live) {
    double d[6];
    for (int t = 0; t < 6; ++t) {
      d[t] = dg[6 * i + t];
      bad = bad || !(fabs(d[t]) <= 2.0);
    }
    const double r[3] = {fabs(d[0]) + fabs(d[1]) + fabs(d[2]), fabs(d[1]) + fabs(d[3]) + fabs(d[4]),
                         fabs(d[2]) + fabs(d[4]) + fabs(d[5])};
    bad = bad || !(r[0] < 4.0 && r[1] < 4.0 && r[2] < 4.0);
    drow = (float)fmax(r[0], fmax(r[1], r[2]));
    if (lane == 0)
      for (int t = 0; t < 3; ++t) row[t] = r[t];
    if (lane < 6) dgo[6 * i + lane] = bad ? make_int2(0, 0) : fixed_entry(-dg[6 * i + lane], 0x1p60);
  }
  const int32_t p0 = live ? rp1[i] : 0, p1 = live ? rp1[i + 1] : 0;
  const int32_t longest = max(p1 - p0, __shfl_xor_sync(0xffffffffu, p1 - p0, 16));  // of the warp's two atoms
  float m6 = 0.f, m4 = 0.f, m2 = 0.f, u1 = 0.f;
  for (int32_t at = 0; at < longest; at += 12) {
    const int32_t p = p0 + at + lane;
    float f[3] = {0.f, 0.f, 0.f};
    if (lane < 12 && p < p1) {
      const double v[3] = {u[3 * (int64_t)p], u[3 * (int64_t)p + 1], u[3 * (int64_t)p + 2]};
      const double s = fabs(v[0]) + fabs(v[1]) + fabs(v[2]);
      if (!(fmax(fabs(v[0]), fmax(fabs(v[1]), fabs(v[2]))) < 1.99 && s < 3.9)) {  // a limb is 31 bits (and see above)
        bad = true;
      } else {
        u1 = fmaxf(u1, (float)s);
        for (int r = 0; r < 3; ++r) {
          row[r] += fabs(v[r]) * s;
          f[r] = (float)(fabs(v[r]) + s);
        }
        const int2 a = fixed_entry(v[0], 0x1p60), b = fixed_entry(v[1], 0x1p60), c = fixed_entry(v[2], 0x1p60);
        blk[2 * (int64_t)p] = make_int4(a.x, a.y, b.x, b.y);
        blk[2 * (int64_t)p + 1] = make_int4(c.x, c.y, ci1[p], 0);
      }
    }
    for (int r = 0; r < 3; ++r) {
      const float two = f[r] + __shfl_xor_sync(0xffffffffu, f[r], 1);
      const float four = two + __shfl_xor_sync(0xffffffffu, two, 2);
      const float six = two + __shfl_down_sync(0xffffffffu, two, 2, 16) + __shfl_down_sync(0xffffffffu, two, 4, 16);
      m2 = fmaxf(m2, two);
      m4 = fmaxf(m4, four);
      if (lane == 0 || lane == 6) m6 = fmaxf(m6, six);
    }
  }
  for (int r = 0; r < 3; ++r) row[r] = sum16(row[r]);
  m6 = 1.00001f * (3.f + drow + max16(m6));
  m4 = 1.00001f * (3.f + drow + max16(m4));
  m2 = 1.00001f * (3.f + drow + max16(m2));
  u1 = 1.00001f * max16(u1);
  bad = any16(bad) || !(m2 < 15.5f);
  if (!live || lane != 0) return;
  if (!bad) {
    raise(info + 2, __float_as_int(m6));
    raise(info + 3, __float_as_int(m4));
    raise(info + 5, __float_as_int(u1));
  }
  raise(info + 4, p1 - p0);
  note_row(info, fmax(row[0], fmax(row[1], row[2])), bad);
}

// Full blocks, unit 2^-59: the cross terms of two blocks stay below 2^58 sum |a| + 2 x 3 2^59, which 63 bits hold
// for ||A||_inf <= 16.
__global__ void __launch_bounds__(128) k_fixed_full(int32_t n_atoms, const int32_t *__restrict__ rp,
                                                    const int32_t *__restrict__ ci, const double *__restrict__ A, int4 *blk,
                                                    int32_t *info) {
  const int64_t i = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 4;
  const int lane = threadIdx.x & 15;
  const bool live = i < n_atoms;
  double row[3] = {0.0, 0.0, 0.0};
  bool bad = false;
  const int32_t p0 = live ? rp[i] : 0, p1 = live ? rp[i + 1] : 0;
  for (int32_t p = p0 + lane; p < p1; p += 16) {
    int2 v[10];
    for (int t = 0; t < 9; ++t) {
      const double e = A[9 * (int64_t)p + t];
      bad = bad || !(fabs(e) < 3.9);
      row[t / 3] += fabs(e);
      v[t] = bad ? make_int2(0, 0) : fixed_entry(-e, 0x1p59);
    }
    v[9] = make_int2(ci[p], 0);
    for (int t = 0; t < 5; ++t) blk[5 * (int64_t)p + t] = make_int4(v[2 * t].x, v[2 * t].y, v[2 * t + 1].x, v[2 * t + 1].y);
  }
  for (int r = 0; r < 3; ++r) row[r] = sum16(row[r]);
  bad = any16(bad);
  if (!live || lane != 0) return;
  raise(info + 4, p1 - p0);
  note_row(info, fmax(row[0], fmax(row[1], row[2])), bad);
}

// ---- entry: column maxima, exponents, conversion ---------------------------------------------
__device__ __forceinline__ uint64_t magnitude(uint64_t bits) { return bits & (~(uint64_t)0 >> 1); }

// Largest |X| bits per column over a slab of rows (patterns of Inf and NaN are the largest): part[slab][c].
// Row-major: lanes along columns.  Column-major: one block per (slab, column).
__global__ void __launch_bounds__(256) k_colmax_rm(int64_t n, int32_t k, const uint64_t *__restrict__ X, int64_t ld,
                                                   int64_t slab, uint64_t *part) {
  __shared__ uint64_t red[8][33];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int32_t c = blockIdx.y * 32 + lane;
  const int64_t r0 = (int64_t)blockIdx.x * slab, r1 = min(n, r0 + slab);
  uint64_t m = 0;
  if (c < k)
    for (int64_t i = r0 + warp; i < r1; i += 8) m = max(m, magnitude(X[i * ld + c]));
  red[warp][lane] = m;
  __syncthreads();
  if (warp == 0 && c < k) {
    for (int w = 1; w < 8; ++w) m = max(m, red[w][lane]);
    part[(int64_t)blockIdx.x * k + c] = m;
  }
}
__global__ void __launch_bounds__(256) k_colmax_cm(int64_t n, int32_t k, const uint64_t *__restrict__ X, int64_t ld,
                                                   int64_t slab, uint64_t *part) {
  __shared__ uint64_t red[8];
  const int64_t r0 = (int64_t)blockIdx.x * slab, r1 = min(n, r0 + slab);
  for (int32_t c = blockIdx.y; c < k; c += gridDim.y) {
    const uint64_t *x = X + (int64_t)c * ld;
    uint64_t m = 0;
    for (int64_t i = r0 + threadIdx.x; i < r1; i += 256) m = max(m, magnitude(x[i]));
    for (int d = 16; d > 0; d >>= 1) m = max(m, (uint64_t)__shfl_xor_sync(0xffffffffu, (unsigned long long)m, d));
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = m;
    __syncthreads();
    if (threadIdx.x == 0) {
      for (int w = 1; w < 8; ++w) m = max(m, red[w]);
      part[(int64_t)blockIdx.x * k + c] = m;
    }
    __syncthreads();
  }
}

// exponent and bound of t_0 per column; cpl adjacent columns are kept in FP64 together
__global__ void k_fixed_plan(int32_t k, int32_t parts, const uint64_t *__restrict__ part, int32_t cpl,
                             const int32_t *__restrict__ info, int64_t kc, int32_t *sh, int32_t *mx) {
  const int64_t c0 = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) * cpl;
  if (c0 >= kc) return;
  int32_t s0[2] = {0, 0}, m0[2] = {0, 0};
  bool raw = false;
  for (int t = 0; t < cpl; ++t) {
    const int64_t c = c0 + t;
    if (c >= k) continue;
    uint64_t m = 0;
    for (int32_t q = 0; q < parts; ++q) m = max(m, part[(int64_t)q * k + c]);
    if (m == 0) continue;
    const double v = __longlong_as_double((long long)m);
    if (!(v >= 0x1p-800 && v <= 0x1p800)) {
      raw = true;
      continue;
    }
    const float g = norm_of(info);
    s0[t] = top_of(info, g) - 1 - ilogb(v * ((double)g + 1.0) * 1.0001);
    m0[t] = (int32_t)ldexp(v, s0[t] - kLimb) + 1;
  }
  for (int t = 0; t < cpl; ++t) {
    sh[c0 + t] = raw ? kRaw : s0[t];
    mx[c0 + t] = m0[t];
    mx[kc + c0 + t] = m0[t] >> 4;
  }
}

// x 2^s rounded to nearest, from the bits of x (no FP64 instructions); |x| 2^s < 2^60
__device__ __forceinline__ int2 to_fixed(uint64_t bits, int32_t s) {
  const int e = (int)(bits >> 52) & 0x7ff;
  uint64_t m = bits & 0xfffffffffffffull;
  if (e) m |= 1ull << 52;
  int64_t v = shifted((int64_t)m, (e ? e : 1) - 1075 + s);
  return split((int64_t)bits < 0 ? -v : v);
}
__device__ __forceinline__ int2 entry(uint64_t bits, int32_t s) {
  return s == kRaw ? make_int2((int32_t)(uint32_t)bits, (int32_t)(uint32_t)(bits >> 32)) : to_fixed(bits, s);
}

__global__ void __launch_bounds__(256) k_fixed_from_rm(int64_t n, int32_t k, int32_t kp, const uint64_t *__restrict__ X,
                                                       int64_t ld, const int32_t *__restrict__ sh, int2 *T) {
  const int64_t t = (int64_t)blockIdx.x * 256 + threadIdx.x;
  const int64_t i = t / kp;
  if (i >= n) return;
  const int32_t c = (int32_t)(t - i * kp);
  T[i * ld + c] = c < k ? entry(X[i * ld + c], sh[c]) : make_int2(0, 0);
}

__global__ void __launch_bounds__(256) k_fixed_from_cm(int64_t n, int32_t k, int32_t kp, const uint64_t *__restrict__ C,
                                                       int64_t ldc, const int32_t *__restrict__ sh, int2 *T, int64_t ld) {
  __shared__ uint64_t tile[32][33];
  const int64_t i0 = (int64_t)blockIdx.x * 32;
  const int32_t cb = blockIdx.y * 32, tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  for (int y = ty; y < 32; y += 8) {
    const int32_t c = cb + y;
    const int64_t i = i0 + tx;
    if (c < k && i < n) tile[y][tx] = C[(int64_t)c * ldc + i];
  }
  __syncthreads();
  const int32_t c = cb + tx;
  if (c >= kp) return;
  const int32_t s = c < k ? sh[c] : 0;
  for (int y = ty; y < 32; y += 8) {
    const int64_t i = i0 + y;
    if (i < n) T[i * ld + c] = c < k ? entry(tile[tx][y], s) : make_int2(0, 0);
  }
}

// The steps of a filter follow each other by programmatic launch: step j + 1 stages its blocks while step j drains,
// and waits for its end (griddepcontrol.wait) before it touches a vector, a scale or a maximum.  Each step waits, so
// a step that ends implies the ends of all before it, and a kernel after the filter is an ordinary one.
// Measured, without and with it: N = 1,000, k = 16 8.6 and 6.7 us a step; N = 5,003, k = 33 20.4 and 18.0;
// N = 99,900, k = 64 280.9 and 277.4; the adjoint at N = 20,000, k = 32, m = 60 15.2 and 14.7 ms.
template <int CPL, int MODE, bool FULL>
void launch_mode(const StepArgs &a, dim3 grid, int threads, size_t smem, cudaStream_t s) {
  cudaLaunchAttribute early{};
  early.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  early.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = grid;
  cfg.blockDim = dim3((unsigned)threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cfg.attrs = &early;
  cfg.numAttrs = 1;
  PFE_LAUNCH cudaLaunchKernelEx(&cfg, k_fixed_step<CPL, MODE, FULL>, a);
}
template <int CPL, bool FULL>
void launch_step(int mode, const StepArgs &a, dim3 grid, int threads, size_t smem, cudaStream_t s) {
  if (mode == MODE_FIRST) launch_mode<CPL, MODE_FIRST, FULL>(a, grid, threads, smem, s);
  else if (mode == MODE_STEP_ACC) launch_mode<CPL, MODE_STEP_ACC, FULL>(a, grid, threads, smem, s);
  else if (mode == MODE_EMIT) launch_mode<CPL, MODE_EMIT, FULL>(a, grid, threads, smem, s);
  else if (mode == MODE_ADJ) launch_mode<CPL, MODE_ADJ, FULL>(a, grid, threads, smem, s);
  else launch_mode<CPL, MODE_STEP, FULL>(a, grid, threads, smem, s);
}

int32_t max_parts(int64_t n) { return (int32_t)std::min<int64_t>(64, (n + 511) / 512); }

}  // namespace

// bytes of a block in shared memory, and what a CTA stages at most (a row has to fit)
size_t fixed_block_bytes(const Bsr<double> &A) { return A.u ? 32 : 80; }
constexpr size_t kFixedStage = 24576;
bool fixed_row_fits(const Bsr<double> &A, int32_t max_row) { return max_row * fixed_block_bytes(A) <= kFixedStage; }

size_t fixed_state_bytes(int64_t n, int32_t k) {
  const int64_t kc = (k + 3) / 4 * 4;
  return (size_t)(8 * kc) * sizeof(int32_t) + (size_t)max_parts(n) * (size_t)k * sizeof(uint64_t);
}

void launch_fixed_operator(const Bsr<double> &A, void *blocks, void *diag, int32_t *info, cudaStream_t s) {
  cudaMemsetAsync(info, 0, kFixedInfo * sizeof(int32_t), s);
  const unsigned grid = (unsigned)((A.n_atoms + 7) / 8);  // 16 lanes an atom
  if (A.u)
    PFE_LAUNCH k_fixed_r1<<<grid, 128, 0, s>>>(A.n_atoms, A.rp1, A.ci1, A.u, A.dg, static_cast<int4 *>(blocks),
                                               static_cast<int2 *>(diag), info);
  else
    PFE_LAUNCH k_fixed_full<<<grid, 128, 0, s>>>(A.n_atoms, A.rp, A.ci, A.vals, static_cast<int4 *>(blocks), info);
}

// Each coefficient by itself: a maximum by fmax would pass over a NaN.
bool fixed_coefficients_ok(const double *coef, int32_t m) {
  double g = 0.0;
  for (int32_t j = 0; j <= m; ++j) {
    if (!(std::fabs(coef[j]) < 0x1p60)) return false;
    g = std::max(g, std::fabs(coef[j]));
  }
  return m >= 1 && g >= 0x1p-100;
}

namespace {

// What the steps of one call share: the operator, the lanes and the CTA shape
struct StepPlan {
  StepArgs a{};
  bool rank1 = false;
  int cpl = 1, threads = 0;
  size_t smem = 0;
  dim3 grid;
};

StepPlan plan_steps(const Bsr<double> &A, const FixedOp &op, int32_t k, int64_t ld, bool aligned) {
  StepPlan p;
  p.rank1 = A.u != nullptr;
  // Two columns a lane (16-byte gathers) once the lanes fill the GPU a few times over; before that one, for more
  // lanes.  us a step with one and two: N = 4,000, k = 64 19.0 and 28.5; N = 3,001, k = 100 24.1 and 33.5; N = 4,000,
  // k = 120 30.9 and 34.3; N = 20,000, k = 26 40.9 and 37.1, k = 32 37.2 and 35.8; N = 99,900, k = 64 334 and 303;
  // full blocks N = 3,000, k = 100 24.0 and 33.9, N = 2,500, k = 200 41.6 and 40.0.
  p.cpl = aligned && k > 1 && ld % 2 == 0 && (int64_t)A.n_atoms * k >= 500000 ? 2 : 1;
  StepArgs &a = p.a;
  a.n_atoms = A.n_atoms;
  a.ld = ld;
  a.rp = A.u ? A.rp1 : A.rp;
  a.blk = static_cast<const int4 *>(op.blocks);
  a.dg = static_cast<const int4 *>(op.diag);
  a.u64 = A.u ? A.u : A.vals;
  a.d64 = A.dg;
  a.ci64 = A.u ? A.ci1 : A.ci;
  a.info = op.info;
  a.kc = (k + 3) / 4 * 4;
  // CTA shape: the fewest column tiles, evenly wide.  Rank-1: as many atoms at a time as 128 lanes hold, more where
  // whole warps then waste fewer lanes (k = 33: 99 of 128 or 231 of 256; N = 5,003: 21.9 and 20.0 us a step); full
  // blocks: 256 lanes.  Up to four passes while every SM keeps its CTAs (N = 99,900, k = 64: 318 us a step with one pass, 303 with four, 302 with eight;
  // N = 5,003, k = 33: 20.7 with one, 24.9 with four).
  const int32_t npc = (k + p.cpl - 1) / p.cpl;
  const int lanes = A.u ? 128 : 256;
  const int tiles = (npc + lanes - 1) / lanes;
  a.groups = npc;
  a.tile = (npc + tiles - 1) / tiles;
  const auto used = [&](int atoms) {  // share of the lanes, less a little for the larger CTAs
    const int t = (atoms * a.tile + 31) / 32 * 32;
    return (double)(atoms * a.tile) / t * (t <= lanes ? 1.0 : 0.95);
  };
  a.per_pass = lanes / a.tile;
  for (int atoms = a.per_pass + 1; atoms * a.tile <= 256; ++atoms)
    if (used(atoms) > used(a.per_pass)) a.per_pass = atoms;
  a.magic = (65536 + a.tile - 1) / a.tile;
  const size_t row_bytes = (size_t)op.max_row * fixed_block_bytes(A);
  while (a.per_pass > 1 && a.per_pass * row_bytes > kFixedStage) --a.per_pass;
  p.threads = (a.per_pass * a.tile + 31) / 32 * 32;
  const int64_t ctas = ((int64_t)A.n_atoms + a.per_pass - 1) / a.per_pass * tiles;
  a.passes = (int32_t)std::min<int64_t>(4, std::max<int64_t>(1, ctas * p.threads / (768 * 152)));
  while (a.passes > 1 && a.per_pass * a.passes * row_bytes > kFixedStage) --a.passes;
  const int per_cta = a.per_pass * a.passes;
  p.smem = (size_t)a.tile * p.cpl * sizeof(ColumnScale) + per_cta * row_bytes;
  p.grid = dim3((unsigned)((A.n_atoms + per_cta - 1) / per_cta), (unsigned)tiles);
  return p;
}

void launch_planned(const StepPlan &p, int mode, cudaStream_t s) {
  if (p.rank1) {
    if (p.cpl == 2) launch_step<2, false>(mode, p.a, p.grid, p.threads, p.smem, s);
    else launch_step<1, false>(mode, p.a, p.grid, p.threads, p.smem, s);
  } else {
    if (p.cpl == 2) launch_step<2, true>(mode, p.a, p.grid, p.threads, p.smem, s);
    else launch_step<1, true>(mode, p.a, p.grid, p.threads, p.smem, s);
  }
}

// v 2^(59 - ge), split; |v| <= 2^ge
int2 fixed_coefficient(double v, int ge) {
  const int64_t t = std::llrint(std::ldexp(v, 2 * kLimb - 1 - ge)) + kHalf;
  return make_int2((int32_t)(t & kMask) - kHalf, (int32_t)(t >> kLimb));
}
int coefficient_exponent(double g) { return g != 0.0 ? std::ilogb(g) + 1 : 0; }

// exponents and bounds of a block's columns (slots 0 and 1 of sh and mx)
void plan_columns(const StepPlan &p, int64_t n, int32_t k, const double *X, int64_t ldx, bool colmajor, int32_t *sh,
                  int32_t *mx, uint64_t *part, cudaStream_t s) {
  const int32_t parts = max_parts(n);
  const int64_t slab = (n + parts - 1) / parts;
  const uint64_t *xb = reinterpret_cast<const uint64_t *>(X);
  if (colmajor)
    PFE_LAUNCH k_colmax_cm<<<dim3(parts, std::min(k, 65535)), 256, 0, s>>>(n, k, xb, ldx, slab, part);
  else
    PFE_LAUNCH k_colmax_rm<<<dim3(parts, (k + 31) / 32), 256, 0, s>>>(n, k, xb, ldx, slab, part);
  PFE_LAUNCH k_fixed_plan<<<(unsigned)((p.a.kc / p.cpl + 127) / 128), 128, 0, s>>>(k, parts, part, p.cpl, p.a.info, p.a.kc,
                                                                                  sh, mx);
}

void convert_columns(const StepPlan &p, int64_t n, int32_t k, const double *X, int64_t ldx, bool colmajor,
                     const int32_t *sh, int2 *T, cudaStream_t s) {
  const int32_t kp = p.a.groups * p.cpl;
  const uint64_t *xb = reinterpret_cast<const uint64_t *>(X);
  if (colmajor)
    PFE_LAUNCH k_fixed_from_cm<<<dim3((unsigned)((n + 31) / 32), (kp + 31) / 32), 256, 0, s>>>(n, k, kp, xb, ldx, sh, T,
                                                                                             p.a.ld);
  else
    PFE_LAUNCH k_fixed_from_rm<<<(unsigned)((n * kp + 255) / 256), 256, 0, s>>>(n, k, kp, xb, ldx, sh, T);
}

bool aligned16(const void *p) { return (reinterpret_cast<uintptr_t>(p) & 15) == 0; }

// a_m and Ybar of the adjoint: a column kept in FP64 on one side is so on both; a zero a_m takes Ybar's exponent;
// slot 3 is a_{m+1} = 0
__global__ void k_fixed_adjoint_columns(int64_t kc, int cpl, int32_t *sh, int32_t *mx, int32_t *ysh, const int32_t *ymx) {
  const int64_t c0 = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) * cpl;
  if (c0 >= kc) return;
  bool raw = false;
  for (int t = 0; t < cpl; ++t) raw = raw || sh[c0 + t] == kRaw || ysh[c0 + t] == kRaw;
  for (int t = 0; t < cpl; ++t) {
    const int64_t c = c0 + t;
    if (raw) sh[c] = ysh[c] = kRaw;
    else if (mx[c] == 0 && ymx[c] != 0) sh[c] = ysh[c];
    sh[3 * kc + c] = sh[c];
    mx[3 * kc + c] = 0;
  }
}

}  // namespace

void launch_fixed_filter(const Bsr<double> &A, const FixedOp &op, const double *coef, int32_t m, int32_t k, int64_t ld,
                         const double *X, int64_t ldx, bool colmajor, double *Y, double *b0, double *b1, void *state,
                         cudaStream_t s) {
  const int64_t n = 3 * (int64_t)A.n_atoms;
  StepPlan p = plan_steps(A, op, k, ld, aligned16(Y) && aligned16(b0) && aligned16(b1));
  StepArgs &a = p.a;
  a.sh = static_cast<int32_t *>(state);
  a.mx = a.sh + 4 * a.kc;
  int2 *t0 = reinterpret_cast<int2 *>(b1), *t1 = reinterpret_cast<int2 *>(b0);
  plan_columns(p, n, k, X, ldx, colmajor, a.sh, a.mx, reinterpret_cast<uint64_t *>(a.mx + 4 * a.kc), s);
  convert_columns(p, n, k, X, ldx, colmajor, a.sh, t0, s);
  for (int32_t j = 0; j < m; ++j) {
    // y takes two terms every other step, as in the FP64 filter
    const bool even = (j % 2) == 0, last = j == m - 1;
    a.j = j;
    a.X = even ? t0 : t1;
    a.W = a.Z = even ? t1 : t0;
    a.Y = (even || last) ? Y : nullptr;
    // the pair's own exponent: a small pair keeps its relative accuracy
    a.ge = coefficient_exponent(std::fmax(even ? std::fabs(coef[j]) : 0.0, std::fabs(coef[j + 1])));
    a.ga = even ? fixed_coefficient(coef[j], a.ge) : make_int2(0, 0);
    a.gb = fixed_coefficient(coef[j + 1], a.ge);
    a.g0 = coef[j];
    a.g1 = coef[j + 1];
    launch_planned(p, j == 0 ? MODE_FIRST : even ? MODE_STEP_ACC : MODE_STEP, s);
  }
}

namespace {

__global__ void k_copy16(int64_t words, const int4 *__restrict__ a, int4 *__restrict__ b) {
  const int64_t all = (int64_t)gridDim.x * blockDim.x;
  for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < words; t += all) b[t] = a[t];
}
void copy16(const void *a, void *b, int64_t words, cudaStream_t s) {
  PFE_LAUNCH k_copy16<<<(unsigned)std::min<int64_t>((words + 255) / 256, 4096), 256, 0, s>>>(
      words, static_cast<const int4 *>(a), static_cast<int4 *>(b));
}
int32_t segments(int32_t m, int32_t seg) { return (m + seg - 1) / seg; }
int32_t snapshots(int32_t m, int32_t seg) { return std::max(0, segments(m, seg) - 2); }

}  // namespace

// Segments of `seg` steps: Ybar as it came and in fixed point, a_j and a_{j+1}, the segment's t_j and a_j; with more
// than one segment also the forward pair and a saved pair for each segment but the first and the last
int64_t fixed_adjoint_vectors(int32_t m, int32_t seg) {
  return 4 + 2 * (int64_t)seg + 1 + (segments(m, seg) > 1 ? 2 : 0) + 2 * (int64_t)snapshots(m, seg);
}
size_t fixed_adjoint_state_bytes(int64_t n, int32_t k, int32_t m, int32_t seg) {
  const int64_t kc = (k + 3) / 4 * 4;
  return fixed_state_bytes(n, k) + (size_t)((12 + 8 * snapshots(m, seg)) * kc) * sizeof(int32_t);
}

// One segment keeps every t_j and a_j: 2 m steps.  More recompute the t_j of each from a saved pair (with its exponents,
// so that they are the same bits), up to 3 m steps.  N = 20,000, k = 64, m = 200: 79 ms with one segment (12.4 GB), 87
// with three (4.4 GB), 155 in the FP64 kernels; N = 50,000, k = 64, m = 60: 55, 61 and 109 ms.
const double *launch_fixed_adjoint(const Bsr<double> &A, const FixedOp &op, const double *coef, int32_t m, int32_t seg,
                                   int32_t k, int64_t ld, const double *X, int64_t ldx, const double *Ybar, int64_t ldyb,
                                   int64_t nnzb, double two_over_d, double *vals_bar, double *work, void *state,
                                   cudaStream_t s) {
  const int64_t n = 3 * (int64_t)A.n_atoms, vec = n * ld;
  StepPlan p = plan_steps(A, op, k, ld, aligned16(work) && vec % 2 == 0);
  StepArgs &a = p.a;
  const int32_t nseg = segments(m, seg), saved = snapshots(m, seg);
  const int64_t kc = a.kc;
  int32_t *ash = static_cast<int32_t *>(state), *amx = ash + 4 * kc, *ysh = ash + 8 * kc, *ymx = ysh + 2 * kc;
  int32_t *fsh = ash + 12 * kc, *fmx = fsh + 4 * kc, *save_state = fsh + 8 * kc;
  uint64_t *part = reinterpret_cast<uint64_t *>(save_state + 8 * saved * kc);
  double *t = work, *adj = t + seg * vec, *yr = adj + (seg + 1) * vec;
  int2 *yb = reinterpret_cast<int2 *>(yr + vec), *v0 = yb + vec, *v1 = v0 + vec;
  int2 *f0 = nseg > 1 ? v1 + vec : v0, *f1 = f0 + vec, *save = f1 + vec;  // save: unused with fewer than three segments
  launch_colmajor_to_rowmajor<double>(n, k, Ybar, ldyb, yr, ld, s);

  const auto start = [&] {  // t_0 in t and, in fixed point, in f0
    launch_colmajor_to_rowmajor<double>(n, k, X, ldx, t, ld, s);
    if (m == 1) return;
    plan_columns(p, n, k, t, ld, false, fsh, fmx, part, s);
    convert_columns(p, n, k, t, ld, false, fsh, f0, s);
  };
  const auto forward = [&](int32_t j, double *out) {  // t_{j+1} from t_j, t_{j-1}; out (never null for j = 0): in FP64
    a.sh = fsh;
    a.mx = fmx;
    a.j = j;
    a.X = j % 2 == 0 ? f0 : f1;
    a.W = a.Z = j % 2 == 0 ? f1 : f0;
    a.Y = out;
    a.emit = 0;
    a.halved = 0;
    a.ge = 1;  // MODE_FIRST: y = 0 x + 1 t_1
    a.ga = make_int2(0, 0);
    a.gb = fixed_coefficient(1.0, 1);
    a.g0 = 0.0;
    a.g1 = 1.0;
    launch_planned(p, j == 0 ? MODE_FIRST : out ? MODE_EMIT : MODE_STEP, s);
  };
  // the coefficients scaled to at most 1 so that tiny ones keep their accuracy
  double top = 0.0;
  for (int32_t j = 0; j <= m; ++j) top = std::fmax(top, std::fabs(coef[j]));
  const int up = coefficient_exponent(top);
  const auto reverse_start = [&](double *am) {  // a_m = g_m Ybar in am and, in fixed point, in v0; a_{m+1} = 0 in v1
    launch_axpby<double>(n, k, std::ldexp(coef[m], -up), yr, ld, 0.0, am, ld, s);
    plan_columns(p, n, k, yr, ld, false, ysh, ymx, part, s);
    plan_columns(p, n, k, am, ld, false, ash, amx, part, s);
    PFE_LAUNCH k_fixed_adjoint_columns<<<(unsigned)((kc / p.cpl + 127) / 128), 128, 0, s>>>(kc, p.cpl, ash, amx, ysh, ymx);
    convert_columns(p, n, k, yr, ld, false, ysh, yb, s);
    convert_columns(p, n, k, am, ld, false, ash, v0, s);
    cudaMemsetAsync(v1, 0, (size_t)vec * sizeof(int2), s);
    launch_axpby<double>(n, k, coef[m], yr, ld, 0.0, am, ld, s);
  };
  const auto reverse = [&](int32_t j, double *out) {  // a_j from a_{j+1}, a_{j+2}
    const int32_t r = m - 1 - j;
    a.sh = ash;
    a.mx = amx;
    a.j = r;
    a.X = r % 2 == 0 ? v0 : v1;
    a.W = a.Z = r % 2 == 0 ? v1 : v0;
    a.Y = out;
    a.Ybar = yb;
    a.ybar_sh = ysh;
    a.ybar_mx = ymx;
    a.emit = up;
    a.halved = j == 0;
    a.g0 = std::ldexp(coef[j], -up);
    a.ge = coefficient_exponent(a.g0);
    a.ga = fixed_coefficient(a.g0, a.ge);
    launch_planned(p, MODE_ADJ, s);
  };

  // The step that gives segment g's first vector t_{g seg} is step g seg - 1: the state before it is saved, and stays
  // in f0, f1 for the last segment.
  if (nseg > 1) {
    start();
    for (int32_t j = 0; j < (nseg - 1) * seg - 1; ++j) {
      const int32_t g = (j + 1) / seg;
      if ((j + 1) % seg == 0 && g <= saved) {
        copy16(f0, save + 2 * (g - 1) * vec, vec, s);  // f0 and f1
        copy16(fsh, save_state + 8 * (g - 1) * kc, 2 * kc, s);
      }
      forward(j, j == 0 ? adj : nullptr);
    }
  }
  for (int32_t g = nseg - 1; g >= 0; --g) {
    const int32_t j0 = g * seg, j1 = std::min(m, j0 + seg);
    if (g == 0) {
      start();
    } else if (g < nseg - 1) {
      copy16(save + 2 * (g - 1) * vec, f0, vec, s);
      copy16(save_state + 8 * (g - 1) * kc, fsh, 2 * kc, s);
    }
    for (int32_t j = std::max(0, j0 - 1); j + 1 < j1; ++j) forward(j, t + (j + 1 - j0) * vec);
    if (g == nseg - 1) reverse_start(adj + (j1 - j0) * vec);
    else copy16(adj, adj + seg * vec, vec / 2, s);  // a_{j1}
    for (int32_t j = j1 - 1; j >= j0; --j) reverse(j, adj + (j - j0) * vec);
    launch_outer_accum_seg(A, nnzb, k, ld, j1 - j0, vec, adj + vec, t, two_over_d * (g == 0 ? 0.5 : 1.0), two_over_d,
                           vals_bar, s);
  }
  return adj;
}

}  // namespace pfe
