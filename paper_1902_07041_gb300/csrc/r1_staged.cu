// The FP32 Chebyshev step on the rank-1 form, with the operator's blocks staged in shared memory.
//
// What bounds it: the gathers of the neighbours' rows.  In the warp-per-row kernel (r1_kernels.cu) each one waits
// for a load of its column index first; here a CTA packs the blocks of its atoms (u, column: 16 bytes each) into
// shared memory, so that the gathers are the loop's only global loads and DEPTH of them are in flight a lane.
// Measured a step, against the warp-per-row kernel at its tuned shape: N = 1,000, k = 16 6.3 -> 3.9 us; N = 20,000,
// k = 1 24.6 -> 9.3, k = 128 34.8 -> 30.1; N = 99,900, k = 64 148 -> 105, k = 128 151 -> 145 (4.2 TB/s of the four
// vector passes), k = 300 425 -> 384, k = 994 1,190 -> 1,140.  At k = 128: three gathers at four CTAs an SM 145 us,
// two 149, one at five CTAs 154.  Narrower tiles for reuse in L1 lose (32 columns 190 us, 64 159).
// Lanes: `tile` column groups of CPL columns times per_pass atoms, so that narrow blocks leave no lanes idle, and
// `passes` atoms one after another a lane.
// The steps follow each other by programmatic launch (see fixed_step.cu): the blocks are staged while the previous
// step drains, and nothing that a step writes is read through the read-only path.
#include "pfe_internal.h"
#include "vec_io.cuh"

namespace pfe {
namespace {

struct StagedArgs {
  int32_t n_atoms;
  int32_t groups, tile;      // CPL-wide column groups per row; of them per CTA
  int32_t per_pass, passes;  // atoms of a CTA at a time, and how often
  uint32_t magic;            // division of a lane's slot by tile: (slot magic) >> 16
  int32_t cap;               // blocks that fit the CTA's shared memory
  int64_t ld;
  const int32_t *rp, *ci;
  const float *u, *dg;
  const float *X, *W;
  float *Z, *Y;
  const float *F, *fs;  // forcing (FORCE): Z += fs[c] F
  float g0, g1;
};

// MODE_FIRST: Z = A X / 2, Y = g0 X + g1 Z;  MODE_STEP: Z = A X - W (+ forcing), Y += g1 Z when given;
// MODE_STEP_ACC: the same with Y += g0 X + g1 Z.  Sums in the order of k_r1_step and k_defect_step: the same results.
template <int CPL, int MODE, bool FORCE, int DEPTH, int MINB>
__global__ void __launch_bounds__(256, MINB) k_r1_staged(const StagedArgs a) {
  extern __shared__ float4 sblk[];
  asm volatile("griddepcontrol.launch_dependents;");
  const uint32_t slot = threadIdx.x, mine = (slot * a.magic) >> 16;
  const int32_t group = blockIdx.y * a.tile + (int32_t)(slot - mine * a.tile);
  const int32_t first = blockIdx.x * (a.per_pass * a.passes), last = min(first + a.per_pass * a.passes, a.n_atoms);
  const int32_t pbase = __ldg(a.rp + first), count = __ldg(a.rp + last) - pbase;
  const bool staged = count <= a.cap;
  const auto block = [&](int32_t p) {  // of the whole list
    const float *u = a.u + 3 * (int64_t)p;
    return make_float4(__ldg(u), __ldg(u + 1), __ldg(u + 2), __int_as_float(__ldg(a.ci + p)));
  };
  if (staged)
    for (int32_t t = threadIdx.x; t < count; t += blockDim.x) sblk[t] = block(pbase + t);
  asm volatile("griddepcontrol.wait;" ::: "memory");
  __syncthreads();
  if ((int32_t)mine >= a.per_pass || group >= a.groups) return;
  const int64_t c0 = (int64_t)group * CPL;
  const uint32_t ldb = (uint32_t)(a.ld * 4), stride = 3 * ldb;
  const char *xl = reinterpret_cast<const char *>(a.X + c0);
  const auto load = [&](int32_t col, float (&x)[3][CPL]) {
    const char *p = xl + (uint64_t)(uint32_t)col * stride;
    ld_n(reinterpret_cast<const float *>(p), x[0]);
    ld_n(reinterpret_cast<const float *>(p + ldb), x[1]);
    ld_n(reinterpret_cast<const float *>(p + 2 * (uint64_t)ldb), x[2]);
  };
  for (int32_t atom = first + (int32_t)mine; atom < last; atom += a.per_pass) {
    float acc[3][CPL];
    {
      const float *d = a.dg + 6 * (int64_t)atom;
      const float dxx = __ldg(d), dxy = __ldg(d + 1), dxz = __ldg(d + 2), dyy = __ldg(d + 3), dyz = __ldg(d + 4),
                  dzz = __ldg(d + 5);
      float x[3][CPL];
      load(atom, x);
#pragma unroll
      for (int c = 0; c < CPL; ++c) {
        acc[0][c] = fmaf(dxx, x[0][c], fmaf(dxy, x[1][c], dxz * x[2][c]));
        acc[1][c] = fmaf(dxy, x[0][c], fmaf(dyy, x[1][c], dyz * x[2][c]));
        acc[2][c] = fmaf(dxz, x[0][c], fmaf(dyz, x[1][c], dzz * x[2][c]));
      }
    }
    const auto add = [&](const float4 &b, const float (&x)[3][CPL]) {
#pragma unroll
      for (int c = 0; c < CPL; ++c) {
        const float s = fmaf(b.x, x[0][c], fmaf(b.y, x[1][c], b.z * x[2][c]));
        acc[0][c] = fmaf(-s, b.x, acc[0][c]);
        acc[1][c] = fmaf(-s, b.y, acc[1][c]);
        acc[2][c] = fmaf(-s, b.z, acc[2][c]);
      }
    };
    int32_t p = __ldg(a.rp + atom) - pbase;
    const int32_t p1 = __ldg(a.rp + atom + 1) - pbase;
    if (staged) {
      for (; p + DEPTH <= p1; p += DEPTH) {
        float x[DEPTH][3][CPL];
#pragma unroll
        for (int v = 0; v < DEPTH; ++v) load(__float_as_int(sblk[p + v].w), x[v]);
#pragma unroll
        for (int v = 0; v < DEPTH; ++v) add(sblk[p + v], x[v]);
      }
      for (; DEPTH > 1 && p < p1; ++p) {
        float x[3][CPL];
        load(__float_as_int(sblk[p].w), x);
        add(sblk[p], x);
      }
    } else {
      for (; p < p1; ++p) {
        const float4 b = block(pbase + p);
        float x[3][CPL];
        load(__float_as_int(b.w), x);
        add(b, x);
      }
    }
    float s[CPL];
    if (FORCE) ldg_n(a.fs + c0, s);
#pragma unroll
    for (int r = 0; r < 3; ++r) {
      const int64_t off = (3 * (int64_t)atom + r) * a.ld + c0;
      float z[CPL], y[CPL], w[CPL], x[CPL], f[CPL];
      const bool with_y = MODE != MODE_STEP || a.Y != nullptr;
      if (MODE != MODE_FIRST) ld_n(a.W + off, w);
      if (FORCE) ldg_n(a.F + off, f);
      if (MODE != MODE_STEP) ld_n(a.X + off, x);
      if (MODE != MODE_FIRST && with_y) ld_n(a.Y + off, y);
#pragma unroll
      for (int c = 0; c < CPL; ++c) {
        z[c] = MODE == MODE_FIRST ? 0.5f * acc[r][c] : acc[r][c] - w[c];
        if (FORCE) z[c] = fmaf(s[c], f[c], z[c]);
        if (MODE == MODE_FIRST) y[c] = fmaf(a.g1, z[c], a.g0 * x[c]);
        else if (MODE == MODE_STEP_ACC) y[c] = fmaf(a.g0, x[c], fmaf(a.g1, z[c], y[c]));
        else y[c] = fmaf(a.g1, z[c], y[c]);
      }
      st_n(a.Z + off, z);
      if (with_y) st_n(a.Y + off, y);
    }
  }
}

bool aligned_to(const void *p, size_t a) { return (reinterpret_cast<uintptr_t>(p) % a) == 0; }

template <int CPL, int MODE, bool FORCE>
void launch_one(const StagedArgs &a, dim3 grid, int threads, size_t smem, cudaStream_t s) {
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
  PFE_LAUNCH cudaLaunchKernelEx(&cfg, k_r1_staged<CPL, MODE, FORCE, 3, 4>, a);
}

template <int CPL>
void launch_cpl(int mode, bool force, const StagedArgs &a, dim3 grid, int threads, size_t smem, cudaStream_t s) {
  if (mode == MODE_FIRST) launch_one<CPL, MODE_FIRST, false>(a, grid, threads, smem, s);
  else if (mode == MODE_STEP_ACC && force) launch_one<CPL, MODE_STEP_ACC, true>(a, grid, threads, smem, s);
  else if (mode == MODE_STEP_ACC) launch_one<CPL, MODE_STEP_ACC, false>(a, grid, threads, smem, s);
  else if (force) launch_one<CPL, MODE_STEP, true>(a, grid, threads, smem, s);
  else launch_one<CPL, MODE_STEP, false>(a, grid, threads, smem, s);
}

}  // namespace

bool r1_staged_usable(const Bsr<float> &A) { return A.u && A.dg && A.rp1 && A.ci1; }

void launch_r1_staged(const Bsr<float> &A, int mode, int32_t k, int64_t ld, const float *X, const float *W, float *Z,
                      float *Y, const float *F, const float *fs, float g0, float g1, cudaStream_t s) {
  if (k <= 0 || A.n_atoms <= 0) return;
  const auto all = [&](size_t b) {
    return aligned_to(X, b) && aligned_to(W, b) && aligned_to(Z, b) && aligned_to(Y, b) && aligned_to(F, b) && aligned_to(fs, b);
  };
  const int cpl = k > 64 && ld % 4 == 0 && all(16) ? 4 : k > 32 && ld % 2 == 0 && all(8) ? 2 : 1;
  StagedArgs a{};
  a.n_atoms = A.n_atoms;
  a.ld = ld;
  a.rp = A.rp1;
  a.ci = A.ci1;
  a.u = A.u;
  a.dg = A.dg;
  a.X = X;
  a.W = W;
  a.Z = Z;
  a.Y = Y;
  a.F = F;
  a.fs = fs;
  a.g0 = g0;
  a.g1 = g1;
  a.groups = (k + cpl - 1) / cpl;
  // Whole rows where 256 lanes hold one, else even tiles: a wide block's gathers then read long runs of memory
  // (N = 99,900: k = 994 1,249 us a step with tiles of 32 groups, 1,195 with 125, 1,140 with whole rows; k = 300
  // 431, 384, 384).  Two passes of narrow tiles (k = 128: 154 us with one, 145 with two, 151 with four), four of wide
  // ones (k = 516: 705 with two, 673 with four), fewer where the CTAs would not fill the GPU.
  const int tiles = (a.groups + 255) / 256;
  a.tile = (a.groups + tiles - 1) / tiles;
  a.per_pass = std::min(256 / a.tile, 128);
  a.magic = (65536 + a.tile - 1) / a.tile;
  const int threads = (a.per_pass * a.tile + 31) / 32 * 32;
  const int64_t ctas = ((int64_t)A.n_atoms + a.per_pass - 1) / a.per_pass * tiles;
  a.passes = (int32_t)std::min<int64_t>(a.tile > 32 ? 4 : 2, std::max<int64_t>(1, ctas / (8 * 152)));
  a.passes = std::min(a.passes, std::max(1, 128 / a.per_pass));
  const int per_cta = a.per_pass * a.passes;
  a.cap = std::min(16 * per_cta + 16, 2560);  // 40 KB at most
  const dim3 grid((unsigned)((A.n_atoms + per_cta - 1) / per_cta), (unsigned)tiles);
  const size_t smem = (size_t)a.cap * sizeof(float4);
  const bool force = F != nullptr;
  if (cpl == 4) launch_cpl<4>(mode, force, a, grid, threads, smem, s);
  else if (cpl == 2) launch_cpl<2>(mode, force, a, grid, threads, smem, s);
  else launch_cpl<1>(mode, force, a, grid, threads, smem, s);
}

}  // namespace pfe
