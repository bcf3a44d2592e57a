// sc_apply_fixed (include/sc.h): q = sum_i scatter_i(F_i gather_i(lambda))
// with the multiply-adds on the integer pipes instead of GB300's narrow FP64
// pipe (paper Eq. "dualop_apply_expl", the per-iteration product).
//
// Per 32x32 stored tile T of F_i and 32-entry block l of lambda:
//   * T is cut to 53-bit fixed point against its largest exponent
//     (M = round(T 2^(52-E)), |T| < 2^E, from the FP64 bit pattern with
//     integer operations), l likewise against its own;
//   * each fixed-point value is split into two 27-bit limbs, M = mh 2^27 + ml;
//   * sum_j M_ij L_j = d2 2^54 + d1 2^27 + d0 with d2 = sum mh lh,
//     d1 = sum (mh ll + ml lh), d0 = sum ml ll: 32x32 -> 64-bit multiply-adds,
//     exact (each term < 2^54, 32 terms < 2^60);
//   * d2, d1, d0 are combined in FP64 and scaled by 2^(E_T + E_l - 2094):
//     one rounding per row and tile.
// Every stored tile is read once from HBM and used for both triangles, as in
// the FP64 apply (rows: lane = row over the tile's columns; columns: lane =
// column over its rows, through the shared-memory copy of the tile).  The
// error is that of representing each tile and lambda block in 53 bits
// relative to their largest entry, about 2^-52 of 32 max|T| max|l| per row
// and tile, the size of an FP64 GEMV's rounding.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>
#include <string>

#include "sc_internal.h"
#include "sc_tiles.cuh"

using namespace sc;

namespace {

constexpr uint32_t kFull = 0xffffffffu;

__device__ __forceinline__ uint32_t exp_field(double x) {
  return (uint32_t)(__double_as_longlong(x) >> 52) & 0x7FFu;
}

// round(x 2^(52 - E)) for |x| < 2^E = 2^(exmax - 1022), split into limbs (hi, lo)
__device__ __forceinline__ int2 fixed_limbs(double x, uint32_t exmax) {
  const uint64_t b = (uint64_t)__double_as_longlong(x);
  const uint32_t ex = (uint32_t)(b >> 52) & 0x7FFu;
  int64_t M = 0;
  if (ex != 0) {
    const uint64_t mant = (b & ((1ull << 52) - 1)) | (1ull << 52);
    const uint32_t s = exmax - ex + 1;            // >= 1
    const uint64_t r = s > 63 ? 0ull : (mant + (1ull << (s - 1))) >> s;
    M = (b >> 63) ? -(int64_t)r : (int64_t)r;
  }
  return make_int2((int)(M & ((1ll << 27) - 1)), (int)(M >> 27));   // (ml, mh)
}

// d2 + d1 2^-27 + d0 2^-54, scaled by 2^e
__device__ __forceinline__ double combine(long long d0, long long d1, long long d2, int e) {
  const double v = fma((double)d0, 0x1p-54, fma((double)d1, 0x1p-27, (double)d2));
  if (e >= -1022 && e <= 1023) return v * __longlong_as_double((long long)(e + 1023) << 52);
  return ldexp(v, e);
}

__device__ __forceinline__ void mac(long long &d0, long long &d1, long long &d2, int2 m, int2 l) {
  // all limbs are exact int32 (|mh|, |lh| <= 2^26, ml, ll < 2^27)
  d0 += (long long)m.x * l.x;
  d1 += (long long)m.y * l.x + (long long)m.x * l.y;
  d2 += (long long)m.y * l.y;
}

constexpr int kStride = 34;                        // doubles between a tile's columns in shared memory (16-byte rows)
constexpr int kApplyWarps = 4;                     // warps per CTA

// In FP64 two stages per warp and 12 warps per SM: a warp's next tile arrives while its multiply-adds hold the
// FP64 pipe (64 heat cubes 197 us, with one stage and 20 warps 203).  In fixed point one stage and 24 warps, whose
// integer chains need the others (64 heat cubes, before the 16-byte accesses below: 146 us and a quarter in FP64 128; 20
// warps 150 and 133; two stages and 12 warps 174 and 158); the limbs of lambda block J lie over the block itself so that six CTAs fit an SM.
// From 64 tiles per resident warp on, the fixed-point runs are handed out in rounds of 32 to 63 tiles: SMs take different
// times for as many tiles, and with one run to a warp all wait for the slowest (512 elasticity cubes 3127 -> 2830 us, 2048
// mixed subdomains 11.25 -> 10.05 ms; 2048 in runs of 128 10.09, of 512 10.77).  FP64 runs gain nothing (4708 us and, in
// runs of 32, 4735 on the 512 cubes).
template <bool kFixed>
struct ApplyShape {
  static constexpr int kStages = kFixed ? 1 : 2, kCtas = kFixed ? 6 : 3;
};

template <int kStages>
struct ApplyWarp {
  double T[kStages][32 * kStride];                 // stages of a tile (column c, row r: c kStride + r)
  union {                                          // lambda block J, in fixed point its limbs
    __align__(16) double pJ[32];
    __align__(16) int2 lJ[32];
  };
  double pI[32];                                   // lambda block I
  __align__(16) int2 lI[32];                       // and its limbs
};

// q += sum of the tiles' products.  The tiles in storage order are cut into one run per warp
// (runs of equal length: the (subdomain, row block) pairs hold 1 .. nt tiles, and a CTA for each left SMs
// waiting), the tiles copied asynchronously; the row block's sum stays in
// registers over its run, the columns' sums are added tile by tile.
// kFixed: of every four tiles of a row block fp64_quarters (0..4) are multiplied in FP64 (FP64 pipe) and the
// rest in fixed point (integer pipes), so that both pipes work at once; else all in FP64.
// Bound by the FP64 pipe (64 multiply-adds of 16 cycles a tile and SM: 173 us for 64 heat cubes), in fixed point by
// integer issue.  Against a CTA per (subdomain, row block), 64 heat cubes (437 MB): FP64 243 -> 199 us, fixed 176 -> 140, a
// quarter in FP64 167 -> 124 (3.5 TB/s); 710 tiles: FP64 31 -> 15 us; 657,000 tiles: FP64 2380 -> 2298, fixed 1569 -> 1407, a
// quarter 1472 -> 1271; 2048 mixed subdomains: 17.3 -> 16.95 ms, 11.2 -> 10.05, 10.5 -> 9.0.
template <bool kFixed>
__global__ void __launch_bounds__(32 * kApplyWarps, ApplyShape<kFixed>::kCtas)
    apply_tiles_kernel(const PlanPtrs P, int64_t n_tasks, int64_t n_tiles, const double *__restrict__ F,
                       const double *__restrict__ lam, double *__restrict__ q, int fp64_quarters) {
  extern __shared__ __align__(16) unsigned char apply_smem[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  constexpr int kStages = ApplyShape<kFixed>::kStages;
  ApplyWarp<kStages> &sm = reinterpret_cast<ApplyWarp<kStages> *>(apply_smem)[warp];
  const int64_t nw = (int64_t)gridDim.x * kApplyWarps, w = (int64_t)blockIdx.x * kApplyWarps + warp;
  const int64_t t0 = n_tiles * w / nw, t1 = n_tiles * (w + 1) / nw;
  if (t0 >= t1) return;
  const bool wide = (reinterpret_cast<uintptr_t>(F) & 15) == 0;   // F is 8-byte aligned, 16 is usual
  auto fetch = [&](int64_t t, int buf) {
    if (!wide) {
      const uint32_t dst = (uint32_t)__cvta_generic_to_shared(&sm.T[buf][lane]);
#pragma unroll 8
      for (int c = 0; c < 32; ++c)
        asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(dst + (uint32_t)(c * kStride * 8)),
                     "l"(F + t * 1024 + c * 32 + lane)
                     : "memory");
      asm volatile("cp.async.commit_group;\n" ::: "memory");
      return;
    }
    const double *src = F + t * 1024 + 2 * lane;   // 16 bytes a lane: two columns to an instruction
    const uint32_t dst = (uint32_t)__cvta_generic_to_shared(&sm.T[buf][(lane >> 4) * kStride + 2 * (lane & 15)]);
#pragma unroll
    for (int c = 0; c < 32; c += 2)
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(dst + (uint32_t)(c * kStride * 8)), "l"(src + c * 32)
                   : "memory");
    asm volatile("cp.async.commit_group;\n" ::: "memory");
  };
  fetch(t0, 0);
  TileCursor cur = tile_at(P, n_tasks, t0);
  const int32_t *map = P.lambda + P.subs[cur.sub].col_off;
  int row = 0, qI = -1;
  uint32_t exI = 0;
  auto load_I = [&]() {                            // lambda block I of the cursor's row block
    row = cur.I * kTile + lane;
    qI = row < cur.m ? map[row] : -1;
    const double p = qI >= 0 ? lam[qI] : 0.0;
    __syncwarp();
    sm.pI[lane] = p;
    if (kFixed) {
      exI = __reduce_max_sync(kFull, exp_field(p));
      sm.lI[lane] = fixed_limbs(p, exI);
    }
  };
  load_I();
  double y = 0.0;
  for (int64_t t = t0; t < t1; ++t) {
    const int buf = (int)(t - t0) % kStages;
    const int J = cur.J, colJ = J * kTile + lane;
    const bool offdiag = J < cur.I;
    const int qJ = colJ < cur.m ? map[colJ] : -1;
    const double p = qJ >= 0 ? lam[qJ] : 0.0;
    if (kStages > 1 && t + 1 < t1) {
      fetch(t + 1, (buf + 1) % kStages);
      asm volatile("cp.async.wait_group 1;\n" ::: "memory");
    } else {
      asm volatile("cp.async.wait_group 0;\n" ::: "memory");
    }
    sm.pJ[lane] = p;
    __syncwarp();
    double *T = sm.T[buf];
    if (!kFixed || J % 4 < fp64_quarters) {        // uniform across the warp
      double y0 = 0.0, y1 = 0.0;                   // the tile's own sum, two chains
#pragma unroll 8
      for (int c = 0; c < 32; c += 2) {
        const double2 l = *reinterpret_cast<const double2 *>(&sm.pJ[c]);
        y0 = fma(T[c * kStride + lane], l.x, y0);
        y1 = fma(T[(c + 1) * kStride + lane], l.y, y1);
      }
      y += y0 + y1;
      if (offdiag) {
        double z0 = 0.0, z1 = 0.0;
#pragma unroll 8
        for (int r = 0; r < 32; r += 2) {
          const double2 v = *reinterpret_cast<const double2 *>(&T[lane * kStride + r]);
          const double2 l = *reinterpret_cast<const double2 *>(&sm.pI[r]);
          z0 = fma(v.x, l.x, z0);
          z1 = fma(v.y, l.y, z1);
        }
        if (qJ >= 0) atomicAdd(q + qJ, z0 + z1);
      }
    } else if constexpr (kFixed) {
      // The cut to fixed point goes entry by entry, so a lane takes the pairs of rows that a 16-byte access holds:
      // half the shared-memory instructions of one entry at a time (512 elasticity cubes, one run to a warp, 3220 -> 3131 us).
      const int e0 = (lane >> 4) * kStride + 2 * (lane & 15);
      uint32_t em = 0;                             // the largest high word holds the largest exponent
#pragma unroll 8
      for (int c = 0; c < 32; c += 2) {
        const double2 v = *reinterpret_cast<const double2 *>(&T[c * kStride + e0]);
        em = max(em, max((uint32_t)__double2hiint(v.x) & 0x7FFFFFFFu, (uint32_t)__double2hiint(v.y) & 0x7FFFFFFFu));
      }
      const uint32_t exT = __reduce_max_sync(kFull, em) >> 20;
      const uint32_t exJ = __reduce_max_sync(kFull, exp_field(p));
      if (exT != 0) {                              // an all-zero tile adds nothing (uniform)
        int2 *Tl = reinterpret_cast<int2 *>(T);    // the limbs in place of the entries
#pragma unroll 8
        for (int c = 0; c < 32; c += 2) {
          const double2 v = *reinterpret_cast<const double2 *>(&T[c * kStride + e0]);
          const int2 x = fixed_limbs(v.x, exT), y1 = fixed_limbs(v.y, exT);
          *reinterpret_cast<int4 *>(&Tl[c * kStride + e0]) = make_int4(x.x, x.y, y1.x, y1.y);
        }
        sm.lJ[lane] = fixed_limbs(p, exJ);
        __syncwarp();
        if (exJ != 0) {
          long long d0 = 0, d1 = 0, d2 = 0, e0 = 0, e1 = 0, e2 = 0;   // two chains each
#pragma unroll 8
          for (int c = 0; c < 32; c += 2) {
            const int4 l = *reinterpret_cast<const int4 *>(&sm.lJ[c]);
            mac(d0, d1, d2, Tl[c * kStride + lane], make_int2(l.x, l.y));
            mac(e0, e1, e2, Tl[(c + 1) * kStride + lane], make_int2(l.z, l.w));
          }
          y += combine(d0 + e0, d1 + e1, d2 + e2, (int)exT + (int)exJ - 2094);
        }
        if (offdiag && exI != 0) {
          long long d0 = 0, d1 = 0, d2 = 0, e0 = 0, e1 = 0, e2 = 0;
#pragma unroll 8
          for (int r = 0; r < 32; r += 2) {
            const int4 v = *reinterpret_cast<const int4 *>(&Tl[lane * kStride + r]);
            const int4 l = *reinterpret_cast<const int4 *>(&sm.lI[r]);
            mac(d0, d1, d2, make_int2(v.x, v.y), make_int2(l.x, l.y));
            mac(e0, e1, e2, make_int2(v.z, v.w), make_int2(l.z, l.w));
          }
          if (qJ >= 0) atomicAdd(q + qJ, combine(d0 + e0, d1 + e1, d2 + e2, (int)exT + (int)exI - 2094));
        }
      }
    }
    __syncwarp();                                  // the next copies overwrite this stage
    if (t + 1 < t1) {
      if (kStages == 1) fetch(t + 1, 0);
      const int sub = cur.sub;
      cur.next(P);
      if (cur.J == 0) {                            // the row block is complete
        if (qI >= 0) atomicAdd(q + qI, y);
        y = 0.0;
        if (cur.sub != sub) map = P.lambda + P.subs[cur.sub].col_off;
        load_I();
      }
    }
  }
  if (qI >= 0) atomicAdd(q + qI, y);
}

// q += the product, launched over all tiles
template <bool kFixed>
cudaError_t launch_tiles(const sc_ctx &c, const double *F, const double *lam, double *q, int fp64_quarters, cudaStream_t st) {
  const int64_t nt = c.sizes.F_doubles / 1024;
  if (nt == 0) return cudaSuccess;
  constexpr int smem = (int)sizeof(ApplyWarp<ApplyShape<kFixed>::kStages>) * kApplyWarps;
  cudaError_t e = cudaFuncSetAttribute(apply_tiles_kernel<kFixed>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e != cudaSuccess) return e;
  int64_t grid = std::min<int64_t>((int64_t)kGridSMs * ApplyShape<kFixed>::kCtas, (nt + kApplyWarps - 1) / kApplyWarps);
  // fixed point: several rounds of runs of 32 to 63 tiles (see ApplyShape)
  if (kFixed) grid *= std::max<int64_t>(1, nt / (kApplyWarps * grid * 32));
  apply_tiles_kernel<kFixed><<<(unsigned)grid, 32 * kApplyWarps, smem, st>>>(c.ptrs(), c.n_apply, nt, F, lam, q,
                                                                           fp64_quarters);
  return cudaGetLastError();
}

}  // namespace

namespace {

sc_status apply_split(sc_ctx *ctx, const double *F_dev, const double *lambda_dev, double *q_dev, int fp64_quarters,
                      void *stream, const char *who) {
  if (!ctx) return SC_ERR_INVALID_ARG;
  if (!ctx->plan_dev && !ctx->blob.empty()) return fail(ctx, SC_ERR_STATE, "sc_upload_plan was not called");
  if (!ctx->has_lambda) return fail(ctx, SC_ERR_STATE, "planned without lambda_map");
  if (ctx->n_dual > 0 && (!lambda_dev || !q_dev)) return fail(ctx, SC_ERR_INVALID_ARG, "lambda_dev or q_dev is NULL");
  if (ctx->sizes.F_doubles > 0 && !F_dev) return fail(ctx, SC_ERR_INVALID_ARG, "F_dev is NULL");
  if (fp64_quarters < 0 || fp64_quarters > 4) return fail(ctx, SC_ERR_INVALID_ARG, "fp64_quarters must be 0..4");
  const cudaStream_t st = static_cast<cudaStream_t>(stream);
  cudaError_t e = cudaSuccess;
  if (ctx->n_dual > 0) e = cudaMemsetAsync(q_dev, 0, sizeof(double) * (size_t)ctx->n_dual, st);
  if (e == cudaSuccess) e = launch_tiles<true>(*ctx, F_dev, lambda_dev, q_dev, fp64_quarters, st);
  if (e != cudaSuccess) return fail(ctx, SC_ERR_CUDA, std::string(who) + ": " + cudaGetErrorString(e));
  return SC_OK;
}

}  // namespace

int sc::launch_apply(const sc_ctx &c, const double *F, const double *lam, double *q, void *stream) {
  return (int)launch_tiles<false>(c, F, lam, q, 4, static_cast<cudaStream_t>(stream));
}

extern "C" sc_status sc_apply_fixed(sc_ctx *ctx, const double *F_dev, const double *lambda_dev, double *q_dev,
                                    void *stream) {
  return apply_split(ctx, F_dev, lambda_dev, q_dev, 0, stream, "sc_apply_fixed");
}

extern "C" sc_status sc_apply_mixed(sc_ctx *ctx, const double *F_dev, const double *lambda_dev, double *q_dev,
                                    int32_t fp64_quarters, void *stream) {
  return apply_split(ctx, F_dev, lambda_dev, q_dev, fp64_quarters, stream, "sc_apply_mixed");
}
