// Split-precision variants of the off-diagonal GEMM work (sm_103a tensor cores).
//
// The paper runs its TRSM/SYRK blocks as FP64 library calls; on GB300 the FP64
// pipe is ~1.2 TFLOP/s while the BF16 tensor path runs at hundreds of TFLOP/s.
// Here the pruned SYRK (paper Sec. 3.3) is computed with an error-free slicing
// of its FP64 operands (the scheme of Ozaki, Ogita, Oishi and Rump, "Error-free
// transformations of matrix multiplication by using fast routines of matrix
// multiplication and its applications", Numer. Algorithms 59, 2012), adapted
// to 8-bit digits:
//
//   * every column j of a subdomain's Y gets one exponent bound 2^Ej over all
//     its rows (|y| < 2^Ej), every row of an L panel block one bound over the
//     block's 32 columns;
//   * |y| 2^-Ej in [0, 1) is cut into S unsigned 8-bit digits u_0..u_{S-1}
//     (y = sign * 2^Ej * sum_t u_t 2^(-8(t+1)) + truncation below 2^(Ej-8S)),
//     taken from the FP64 bit pattern with integer operations only; each
//     signed digit is exactly a BF16 value;
//   * products of digit planes t and t' run on the tensor cores (mma.sync
//     m16n8k16, BF16 in, FP32 accumulate); for one 32-row block the sum over
//     all pairs with t + t' = d is an integer below 7 * 32 * 255^2 < 2^24, so
//     the FP32 accumulator holds it exactly;
//   * the exact block sums are added as int32 (flushed every 128 blocks), the
//     digit groups are combined exactly in 64-bit integers, and the output
//     sum_d I_d 2^(-8(d+2)) * 2^(Ej1 + Ej2) is formed with one conversion to
//     FP64 and one scaling (the FP64 pipe is the scarce resource on GB300).
//
// L and Y are cut into digit planes once per assembly (lpack_kernel after
// the reciprocal diagonal; yslice after the TRSM, which leaves Y's column bounds), so the TRSM and
// SYRK tasks only load BF16 planes.
//
// Only pairs with t + t' <= S - 1 are formed (S(S+1)/2 products); the terms
// dropped and the digit truncation are below 2^(-8S) relative to the
// product of the column bounds.  S = 7 keeps 56 bits of every operand.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>

#include "sc_digits.cuh"
#include "sc_internal.h"
#include "sc_trsm.cuh"

namespace sc {

namespace {

using namespace digits;

constexpr int kPad = 40;   // bf16 row stride of a digit plane (conflict-free fragment loads)

__device__ __forceinline__ void mma_bf16(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
      "{%0,%1,%2,%3};\n"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

__device__ __forceinline__ uint32_t ld_pair(const __nv_bfloat16 *p) {
  return *reinterpret_cast<const uint32_t *>(p);
}

// Digit planes of L's panel rows below one 32x32 diagonal block (one CTA per
// (supernode, block) item; one thread per panel row, so every CSC column is
// read contiguously).  The 16 words of a plane's row are stored word w at 4 (w mod 4) + w / 4: the four that a lane
// of the update needs are then one 16-byte load.  Blocks of up to kDirect columns need no planes.
template <int S>
__global__ void __launch_bounds__(kThreads) lpack_kernel(const PlanPtrs P, const double *__restrict__ Lv,
                                                         __nv_bfloat16 *__restrict__ Ld,
                                                         int16_t *__restrict__ lexp, int64_t ld_rows) {
  const int si = P.sblk[2 * blockIdx.x], b = P.sblk[2 * blockIdx.x + 1];
  const SnDev s = P.sns[si];
  const int64_t *cp = P.lcp + s.lcp_off;
  const int nrow = s.ns + s.rs;
  const int kb = 32 * b, kw = min(32, s.ns - kb);
  const int nb = nrow - kb - kw;
  if (kw <= kDirect) return;
  const int64_t base = s.ld_off + (int64_t)b * nrow - 16LL * b * (b + 1);
  for (int r = threadIdx.x; r < nb; r += kThreads) {
    const int p = kb + kw + r;
    double v[32];
    int e = 0;
#pragma unroll
    for (int q = 0; q < 32; ++q) {
      v[q] = q < kw ? Lv[cp[kb + q] - (kb + q) + p] : 0.0;
      e = max(e, biased_exponent(v[q]));
    }
    lexp[base + r] = (int16_t)e;
    uint64_t X[32];
    uint32_t neg = 0;
#pragma unroll
    for (int q = 0; q < 32; ++q) {
      X[q] = fixed_point(v[q], e);                  // once per entry, not once per digit plane
      neg |= (v[q] < 0.0 ? 1u : 0u) << q;
    }
#pragma unroll
    for (int d = 0; d < S; ++d) {
      // the row's 64 bytes of this plane as four 16-byte stores
      uint4 *row = reinterpret_cast<uint4 *>(Ld + (int64_t)d * ld_rows * 32 + (base + r) * 32);
#pragma unroll
      for (int g = 0; g < 4; ++g) {
        uint32_t w[4];
#pragma unroll
        for (int h = 0; h < 4; ++h) {
          const int q = 2 * (4 * h + g);          // word 4 h + g of the row
          const __nv_bfloat16 lo = digit_bf16(X[q], d, (neg >> q) & 1u);
          const __nv_bfloat16 hi = digit_bf16(X[q + 1], d, (neg >> (q + 1)) & 1u);
          w[h] = (uint32_t)__bfloat16_as_ushort(lo) | ((uint32_t)__bfloat16_as_ushort(hi) << 16);
        }
        row[g] = make_uint4(w[0], w[1], w[2], w[3]);
      }
    }
  }
}

// Digit planes of Y for one (supernode, 32-row block) item: 32x32 tiles are
// read row-wise (coalesced), transposed in shared memory and written
// column-major (coalesced), rows padded to 32.
// kBalanced (the tcgen05 SYRK's planes): the magnitude is cut against twice the
// column bound (|y| 2^-(Ej + 1) < 1/2, so the top digit is at most 127) and
// recoded into balanced digits in [-128, 128] (least significant first: a
// digit above 127 becomes digit - 256 and carries one into the next), so
// every digit product is at most 2^14 in magnitude.
template <int S, bool kBalanced>
__global__ void __launch_bounds__(kThreads) yslice_kernel(const PlanPtrs P, const double *__restrict__ Y,
                                                          const int *__restrict__ colexp,
                                                          __nv_bfloat16 *__restrict__ Yd, int64_t yd_plane) {
  __shared__ double Ts[32][33];
  const int si = P.sblk[2 * blockIdx.x], b = P.sblk[2 * blockIdx.x + 1];
  const SnDev s = P.sns[si];
  const SubDev sd = P.subs[s.sub];
  const int ws = s.jhi - s.jlo;
  const int npad = (s.ns + 31) / 32 * 32;
  const int r0 = 32 * b;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int c0 = 0; c0 < ws; c0 += 32) {
    for (int i = warp; i < 32; i += kThreads / 32) {
      const int r = r0 + i, c = c0 + lane;
      Ts[i][lane] = (r < s.ns && c < ws) ? Y[s.y_off + (int64_t)r * ws + c] : 0.0;
    }
    __syncthreads();
    for (int j = warp; j < 32; j += kThreads / 32) {
      const int c = c0 + j;
      if (c < ws) {
        const double v = Ts[lane][j];
        const int64_t e = s.yd_off + (int64_t)c * npad + r0 + lane;
        if (kBalanced) {
          const uint64_t X = fixed_point(v, colexp[sd.col_off + s.jlo + c] + 1);
          int dig[S];
          int carry = 0;
#pragma unroll
          for (int d = S - 1; d >= 0; --d) {
            int u = (int)((X >> (55 - 8 * d)) & 0xFF) + carry;
            carry = (d > 0 && u >= 128) ? 1 : 0;
            dig[d] = u - 256 * carry;
          }
#pragma unroll
          for (int d = 0; d < S; ++d)
            Yd[(int64_t)d * yd_plane + e] = __float2bfloat16_rn(v < 0.0 ? -(float)dig[d] : (float)dig[d]);
        } else {
          const uint64_t X = fixed_point(v, colexp[sd.col_off + s.jlo + c]);
#pragma unroll
          for (int d = 0; d < S; ++d) Yd[(int64_t)d * yd_plane + e] = digit_bf16(X, d, v < 0.0);
        }
      }
    }
    __syncthreads();
  }
}

constexpr int kSyrkBatch = 64;   // supernodes whose rows are numbered through at a time

// Y's digit rows that are live on a task's chunks, in units of 8 (a 16-byte copy per column and plane)
struct SyrkUnits {
  int64_t off[kSyrkBatch];             // digit offset of (first live row, sorted column 0)
  int start[kSyrkBatch + 1];           // first unit of every supernode of the batch
  int npad[kSyrkBatch], jlo[kSyrkBatch], jhi[kSyrkBatch];
  int wsum;
};

__device__ __forceinline__ void ldmatrix_x4(uint32_t (&r)[4], const __nv_bfloat16 *p) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];\n"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"((uint32_t)__cvta_generic_to_shared(p)));
}

// One 32x32 block of F = Y^T Y (sorted chunks q1 >= q2) from Y's digit
// planes.  Warp w computes rows 16*(w>>1).. and columns 16*(w&1).. of the
// block as two m16n8 tiles.  The live rows of all listed supernodes are numbered
// through in units of 8 and taken four units at a time (K = 32), whatever
// supernodes they belong to; the next four are copied asynchronously meanwhile.
// Bound by mma.sync issue (2.3 ms for 64 heat cubes at 7 digits).  Against one stage per supernode block and
// word loads of the fragments, SYRK with its slicing, 7 digits: 64 heat cubes 5.84 -> 5.15 ms, 8
// elasticity cubes 1.15 -> 1.08 ms, 36 squares 328 -> 135 us, one square 140 -> 41 us.
template <int S>
// 4 resident CTAs for up to 5 digits, 3 for 6 and 7 (register-bound fragments)
__global__ void __launch_bounds__(kThreads, (S <= 5 ? 4 : 3)) syrk_split_kernel(const PlanPtrs P, const __nv_bfloat16 *__restrict__ Yd,
                                                              int64_t yd_plane, const int *__restrict__ colexp,
                                                              double *__restrict__ F) {
  // two stages of the digit tiles: [stage][operand][t][column][k]
  extern __shared__ __align__(16) unsigned char syrk_smem[];
  typedef __nv_bfloat16 Tile[S][32][kPad];
  Tile *stages = reinterpret_cast<Tile *>(syrk_smem);          // stages[2 * buf + op]
  __shared__ SyrkUnits un;
  const SyrkTask t = P.syrk_tasks[blockIdx.x];
  const SubDev sd = P.subs[t.sub];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int g = lane >> 2, tg = lane & 3;
  const int j1lo = t.q1 * kChunk, j2lo = t.q2 * kChunk;
  const int mrow = 16 * (warp >> 1), ncol = 16 * (warp & 1);
  // per output: the Horner words of the digit-group sums, accumulated over
  // stages (linear, exact: < 128 stages * 2^24 * 256^(h-1) < 2^63)
  Groups<S> acc[8];
  double dacc[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) dacc[i] = 0.0;
  int blocks = 0;
  for (int l0 = 0; l0 < t.list_len; l0 += kSyrkBatch) {
    int n = 0;
    if (tid < kSyrkBatch && l0 + tid < t.list_len) {
      const SnDev s = P.sns[P.syrk_list[t.list_off + l0 + tid]];
      const int nb = (s.ns + 31) >> 5;
      int b = 0;
      while (b < nb && P.cuts[s.cut_off + b] <= j1lo) ++b;     // rows before the first live block are zero on q1
      n = max(0, s.ns - 32 * b + 7) >> 3;
      const int npad = 32 * nb;
      un.npad[tid] = npad;
      un.off[tid] = s.yd_off - (int64_t)s.jlo * npad + 32 * b;
      un.jlo[tid] = s.jlo;
      un.jhi[tid] = s.jhi;
    }
    int inc = n;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const int v = __shfl_up_sync(0xffffffffu, inc, d);
      if (lane >= d) inc += v;
    }
    if (tid == 31) un.wsum = inc;
    __syncthreads();
    if (tid < kSyrkBatch) un.start[tid + 1] = inc + (warp == 1 ? un.wsum : 0);
    if (tid == 0) un.start[0] = 0;
    __syncthreads();
    const int total = un.start[kSyrkBatch];
    // this thread copies unit `part` of column `col` of every stage, all planes of both operands
    const int part = tid & 3, col = tid >> 2;
    auto fetch = [&](int st) {
      const int u = 4 * st + part;
      const __nv_bfloat16 *src[2] = {Yd, Yd};
      int bytes[2] = {0, 0};
      if (u < total) {
        int e = 0;
#pragma unroll
        for (int h = kSyrkBatch / 2; h >= 1; h >>= 1)
          if (un.start[e + h] <= u) e += h;
        const int64_t off = un.off[e] + 8 * (u - un.start[e]);
#pragma unroll
        for (int op = 0; op < 2; ++op) {
          const int j = (op == 0 ? j1lo : j2lo) + col;
          if (j >= un.jlo[e] && j < un.jhi[e]) {
            src[op] = Yd + off + (int64_t)j * un.npad[e];
            bytes[op] = 16;
          }
        }
      }
#pragma unroll
      for (int op = 0; op < 2; ++op) {
        const uint32_t dst = (uint32_t)__cvta_generic_to_shared(&stages[2 * (st & 1) + op][0][col][8 * part]);
        const int64_t step = bytes[op] ? yd_plane : 0;
#pragma unroll
        for (int d = 0; d < S; ++d)
          asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(dst + (uint32_t)(d * 32 * kPad * 2)),
                       "l"(src[op] + d * step), "r"(bytes[op])
                       : "memory");
      }
      asm volatile("cp.async.commit_group;\n" ::: "memory");
    };
    const int nst = (total + 3) >> 2;
    if (nst > 0) fetch(0);
    for (int st = 0; st < nst; ++st) {
      if (st + 1 < nst) {
        fetch(st + 1);
        asm volatile("cp.async.wait_group 1;\n" ::: "memory");   // this stage's copies are done
      } else {
        asm volatile("cp.async.wait_group 0;\n" ::: "memory");
      }
      __syncthreads();
      const Tile &PA = stages[2 * (st & 1)], &PB = stages[2 * (st & 1) + 1];
      // rows of the fragments that this lane's ldmatrix address names
      const int ar = mrow + (lane & 15), ak = 8 * (lane >> 4);
      const int br = ncol + (lane & 7) + 8 * (lane >> 4), bk = 8 * ((lane >> 3) & 1);
#pragma unroll
      for (int d = 0; d < S; ++d) {
        float c[2][4] = {{0.f, 0.f, 0.f, 0.f}, {0.f, 0.f, 0.f, 0.f}};
#pragma unroll
        for (int ta = 0; ta <= d; ++ta) {
          const int tb = d - ta;
#pragma unroll
          for (int ks = 0; ks < 32; ks += 16) {
            uint32_t a[4], b[4];
            ldmatrix_x4(a, &PA[ta][ar][ks + ak]);
            ldmatrix_x4(b, &PB[tb][br][ks + bk]);
            mma_bf16(c[0], a, b[0], b[1]);
            mma_bf16(c[1], a, b[2], b[3]);
          }
        }
#pragma unroll
        for (int nt = 0; nt < 2; ++nt)
#pragma unroll
          for (int r = 0; r < 4; ++r) acc[nt * 4 + r].accumulate(d, __float2int_rn(c[nt][r]));
      }
      __syncthreads();                // the next fetch overwrites this stage (or the next batch the units)
      if (++blocks == 128) {          // int64 headroom, see acc
        blocks = 0;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          dacc[i] += acc[i].value_wide();
          acc[i] = Groups<S>();
        }
      }
    }
  }
  const int32_t *perm = P.perm_cols + sd.col_off;
  const int *ce = colexp + sd.col_off;
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const int nt = i >> 2, r = i & 3;
    const int rl = mrow + g + ((r & 2) ? 8 : 0);
    const int cl = ncol + 8 * nt + 2 * tg + (r & 1);
    const int j1 = j1lo + rl, j2 = j2lo + cl;
    if (j1 < sd.m && j2 < sd.m && (t.q1 != t.q2 || j1 >= j2)) {
      double v = dacc[i] + acc[i].value_wide();
      const int e = (ce[j1] - 1022) + (ce[j2] - 1022);
      v = (e >= -1022 && e <= 1023) ? v * pow2i(e) : ldexp(v, e);
      const int a = perm[j1], b = perm[j2];
      const int hi = max(a, b), lo = min(a, b);
      const int I = hi / kTile, J = lo / kTile;
      double *T = F + sd.F_off + ((int64_t)I * (I + 1) / 2 + J) * (kTile * kTile);
      T[(hi % kTile) + kTile * (lo % kTile)] = v;
      if (I == J) T[(lo % kTile) + kTile * (hi % kTile)] = v;
    }
  }
}

// ---- sparse TRSM with split-precision updates ------------------------------
//
// A CTA of four warps has 4 C columns of a 32-column chunk, C to a warp.  A warp
// solves the triangles of its own columns in FP64 (sc_trsm.cuh), without waiting
// for the others; the update of the rows below a block of more than kDirect columns
// is the CTA's: its columns' digit planes in shared memory, the rows' m-tiles dealt to the
// warps, each L fragment used for all of the CTA's columns.  Narrow CTAs (C = 2) have
// the shorter triangles and fill the GPU on small batches; C is chosen as the FP64 TRSM's
// columns per warp are (sc_plan.cpp).  Batches of large subdomains take trsm_chunk_kernel below.  Bound by the FP64 pipe (triangles, and two
// operations per entry and block after the digit products) and by latency.  Against one CTA
// per 32-column chunk whose warps shared each triangle 8 columns at a time, 7 digits, TRSM with its packing:
// one square 312 -> 64 us, 36 squares 1.11 -> 0.33 ms, 8 elasticity cubes 4.04 -> 2.31 ms.

struct TrsmSplit {
  const __nv_bfloat16 *Ld;     // digit planes of L
  const int16_t *lexp;         // its rows' exponent bounds
  int64_t ld_rows;
  int *colexp;                 // exponent bounds of Y's columns (out)
  const unsigned *unscaled;    // not 0: triangles are not divided by their diagonal (prep_kernel)
};

// A lane's fragments of the S digit planes of L, panel rows row (va) and row + 8 (vb): by words, which arrive where the
// products need them, or (kVector) by 16-byte loads, a quarter of the loads, but their registers have to be regrouped for
// every product.  By words / by vectors, TRSM with packing at 7 digits: 64 heat cubes 5.9 / 6.3 ms with 4 columns to a warp,
// 5.3 / 6.2 with the whole chunk on a CTA; at 5 digits and below, and with 2 columns to a warp (8 elasticity cubes
// 2.41 / 2.33), where the registers suffice for both, the vectors are as fast or faster.
template <int S, bool kVector>
struct Fragments;
template <int S>
struct Fragments<S, false> {
  uint32_t w[S][2][4];
  __device__ __forceinline__ void load(const TrsmSplit &sp, int64_t row, bool va, bool vb, int tg) {
#pragma unroll
    for (int d = 0; d < S; ++d) {
      const uint32_t *pw = reinterpret_cast<const uint32_t *>(sp.Ld + (int64_t)d * sp.ld_rows * 32) + row * 16 + 4 * tg;
#pragma unroll
      for (int ks = 0; ks < 2; ++ks) {
        w[d][ks][0] = va ? pw[2 * ks] : 0u;
        w[d][ks][1] = vb ? pw[128 + 2 * ks] : 0u;
        w[d][ks][2] = va ? pw[2 * ks + 1] : 0u;
        w[d][ks][3] = vb ? pw[128 + 2 * ks + 1] : 0u;
      }
    }
  }
  // c += (the rows' plane d) (the column of X's digits at px)
  __device__ __forceinline__ void mma(float (&c)[4], int d, const __nv_bfloat16 *px) const {
    mma_bf16(c, w[d][0], ld_pair(px), ld_pair(px + 8));
    mma_bf16(c, w[d][1], ld_pair(px + 16), ld_pair(px + 24));
  }
};
template <int S>
struct Fragments<S, true> {
  uint4 a[S], b[S];
  __device__ __forceinline__ void load(const TrsmSplit &sp, int64_t row, bool va, bool vb, int tg) {
#pragma unroll
    for (int d = 0; d < S; ++d) {
      const uint4 *pl = reinterpret_cast<const uint4 *>(sp.Ld + (int64_t)d * sp.ld_rows * 32) + row * 4 + tg;
      a[d] = va ? pl[0] : make_uint4(0u, 0u, 0u, 0u);
      b[d] = vb ? pl[32] : make_uint4(0u, 0u, 0u, 0u);
    }
  }
  __device__ __forceinline__ void mma(float (&c)[4], int d, const __nv_bfloat16 *px) const {
    const uint32_t w0[4] = {a[d].x, b[d].x, a[d].y, b[d].y};
    const uint32_t w1[4] = {a[d].z, b[d].z, a[d].w, b[d].w};
    mma_bf16(c, w0, ld_pair(px), ld_pair(px + 8));
    mma_bf16(c, w1, ld_pair(px + 16), ld_pair(px + 24));
  }
};

template <int C, int S>
struct TeamShared {
  TrsmShared<C> w[kThreads / 32];
  double T[32 * 31 / 2];                            // a wide block's triangle over its diagonal, L(row, p) / L(p, p)
  __align__(16) __nv_bfloat16 PX[S][4 * C][kPad];   // digit planes of the block's X: [digit][live column][row]
  int emax[4 * C];                                  // and their columns' exponent bounds
};

template <int C, int S>
__device__ __forceinline__ void trsm_team(const PlanPtrs &P, const TrsmTask &t, int part, const double *__restrict__ Lv,
                                          const double *__restrict__ invd, const TrsmSplit &sp,
                                          double *__restrict__ Y, TeamShared<C, S> &sm, int warp, int lane) {
  constexpr int kRows = 32 / C;                                    // rows of a block's X that a warp's lanes cover
  const int g = lane >> 2, tg = lane & 3;
  const int c_lo = t.c_lo + part * 4 * C, c_hi = min(c_lo + 4 * C, t.c_lo + t.w);
  if (c_lo >= c_hi) return;                                        // uniform
  const int w_lo = min(c_lo + warp * C, c_hi), w_hi = min(w_lo + C, c_hi);   // this warp's columns
  TrsmShared<C> &own = sm.w[warp];
  int *colexp = sp.colexp + P.subs[t.sub].col_off;
  int n = 0;
  for (int l0 = 0; l0 < t.list_len; l0 += 32) {
    n = trsm_batch(P, t, l0, c_lo, c_hi, own.sn, lane);
    for (int i = 0; i < n; ++i) {
      const TrsmSn &s = own.sn[i];
      const int j = w_lo + lane % C, ws = s.jhi - s.jlo;
      if (j >= s.jlo && j < min(s.jhi, w_hi))
        for (int r = lane / C; r < s.ns; r += kRows) Y[s.y_off + (int64_t)r * ws + j - s.jlo] = 0.0;
    }
  }
  __syncwarp();
  {
    const int32_t *seed = P.seed_ptr + P.subs[t.sub].col_off;
    const int e1 = seed[w_hi];
    for (int e = seed[w_lo] + lane; e < e1; e += 32) Y[P.seeds[e].y_off] = P.seeds[e].value;
  }
  __syncwarp();

  for (int l0 = 0; l0 < t.list_len; l0 += 32) {
    if (t.list_len > 32) n = trsm_batch(P, t, l0, c_lo, c_hi, own.sn, lane);
    for (int i = 0; i < n; ++i) {
      const TrsmSn s = own.sn[i];
      const int ws = s.jhi - s.jlo, nr = s.ns + s.rs;
      const int a4 = max(s.jlo, c_lo), b4 = min(s.jhi, c_hi);      // the CTA's live columns
      const int a = max(s.jlo, w_lo), b = min(s.jhi, w_hi);        // the warp's
      const int64_t *rm = P.rmap + s.rmap_off;
      const double *Lc = Lv + s.lval;
      for (int kb = 0, blk = 0; kb < s.ns; kb += 32, ++blk) {
        const int kw = min(32, s.ns - kb), below = kb + kw, nb = nr - below;
        const int cut = P.cuts[s.cut_off + blk];
        const int wk4 = min(b4, cut) - a4, wk = min(b, cut) - a;
        if (wk4 > 0) {                                             // uniform
          const bool team = kw > kDirect && nb > 0;
          double *Ys = Y + s.y_off + (a - s.jlo);
          int em = 0;
          const double idv = lane < kw ? invd[s.lcp_off + kb + lane] : 0.0;
          if (kw > kDirect) {                                      // the CTA's warps share the triangle
#pragma unroll 4
            for (int p = warp; p < kw; p += kThreads / 32) {
              const double inv = __shfl_sync(0xffffffffu, idv, p);
              // panel row kb + lane of column kb + p
              if (lane > p && lane < kw) sm.T[tri_at(lane, p)] = Lc[kb + lane + p * (nr - kb - 1) - p * (p - 1) / 2] * inv;
            }
            __syncthreads();
          }
          if (wk > 0) {
            if (kw > kDirect) {
              trsm_triangle<C, true>(own, sm.T, Ys + (int64_t)kb * ws, ws, kw, wk, idv, lane);
            } else {
              trsm_stage_triangle(own, Lc, nr, kb, kw, lane);
              asm volatile("cp.async.wait_group 0;\n" ::: "memory");
              __syncwarp();
              trsm_triangle<C, false>(own, own.T, Ys + (int64_t)kb * ws, ws, kw, wk, idv, lane);
            }
            __syncwarp();
            // the columns' exponent bounds, for the digits of X and for Y's planes
            if (lane % C < wk)
              for (int r = lane / C; r < kw; r += kRows) em = max(em, biased_exponent(own.X[r][lane % C]));
#pragma unroll
            for (int d = C; d < 32; d <<= 1) em = max(em, __shfl_xor_sync(0xffffffffu, em, d));
            if (lane < wk && em) atomicMax(colexp + a + lane, em);
          }
          if (team) {
            if (wk > 0) {
              const int cl = lane % C, cc = a - a4 + cl;
              if (lane < wk) sm.emax[cc] = em;
              if (cl < wk)
                for (int r = lane / C; r < 32; r += kRows) {
                  const double v = r < kw ? own.X[r][cl] : 0.0;
                  const uint64_t m = fixed_point(v, em);
#pragma unroll
                  for (int d = 0; d < S; ++d) sm.PX[d][cc][r] = digit_bf16(m, d, v < 0.0);
                }
            }
            __syncthreads();
            const int64_t base = s.ld_off + (int64_t)blk * nr - 16LL * blk * (blk + 1);
            const int colsh = a4 - s.jlo;
            for (int r0 = 16 * warp; r0 < nb; r0 += 16 * (kThreads / 32)) {
              const int ra = r0 + g, rb = r0 + g + 8;
              const bool va = ra < nb, vb = rb < nb;
              Fragments<S, (C < 4 || S <= 5)> fr;
              fr.load(sp, base + ra, va, vb, tg);
              const int ea = va ? sp.lexp[base + ra] : 0, eb = vb ? sp.lexp[base + rb] : 0;
              double *ta = nullptr, *tb = nullptr;                 // this lane's two target rows
              if (va) ta = Y + colsh + (below + ra < s.ns ? s.y_off + (int64_t)(below + ra) * ws : rm[below + ra - s.ns]);
              if (vb) tb = Y + colsh + (below + rb < s.ns ? s.y_off + (int64_t)(below + rb) * ws : rm[below + rb - s.ns]);
#pragma unroll
              for (int nt = 0; nt < C / 2; ++nt) {
                if (8 * nt >= wk4) break;                          // uniform
                // the targets' current values, loaded before the products so that
                // their latency overlaps the MMAs
                double yv[4];
#pragma unroll
                for (int r = 0; r < 4; ++r) {
                  const int col = 8 * nt + 2 * tg + (r & 1);
                  const double *p = (r & 2) ? tb : ta;
                  yv[r] = (p && col < wk4) ? p[col] : 0.0;
                }
                Groups<S> gr[4];
#pragma unroll
                for (int d = 0; d < S; ++d) {
                  float c[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
                  for (int q = 0; q <= d; ++q) {
                    const __nv_bfloat16 *px = &sm.PX[d - q][8 * nt + g][2 * tg];
                    fr.mma(c, q, px);
                  }
#pragma unroll
                  for (int r = 0; r < 4; ++r) gr[r].add(d, __float2int_rn(c[r]));
                }
#pragma unroll
                for (int r = 0; r < 4; ++r) {
                  const int col = 8 * nt + 2 * tg + (r & 1);
                  double *p = (r & 2) ? tb : ta;
                  if (p && col < wk4) {
                    // one conversion and one FMA on the FP64 pipe: both power-of-two
                    // scalings folded into a single exponent
                    const int e = ((r & 2 ? eb : ea) - 1022) + (sm.emax[col] - 1022) + Groups<S>::kBlockShift;
                    const double v = (double)gr[r].block_int();
                    p[col] = (e >= -1022 && e <= 1023) ? fma(-v, pow2i(e), yv[r]) : yv[r] - ldexp(v, e);
                  }
                }
              }
            }
            __syncthreads();
          } else if (kw > kDirect) {
            __syncthreads();                                       // T is read by all
          } else if (wk > 0) {
            // FP64 update of the warp's own columns: (row, column) pairs, four to a lane
            const int dp = 32 / wk, cl = lane % wk;
            for (int p0 = below + (lane < dp * wk ? lane / wk : nr); __any_sync(0xffffffffu, p0 < nr); p0 += 4 * dp) {
              int row[4];
              const int col[4] = {cl, cl, cl, cl};
              double *tg4[4];
              double acc[4];
              int last = 0;
#pragma unroll
              for (int j = 0; j < 4; ++j) {
                const int p = p0 + j * dp;
                const bool ok = p < nr;
                if (__any_sync(0xffffffffu, ok)) last = j + 1;
                row[j] = ok ? p : nr - 1;
                tg4[j] = !ok ? nullptr : (p < s.ns ? Ys + (int64_t)p * ws : Y + rm[p - s.ns] + (a - s.jlo)) + cl;
                acc[j] = ok ? *tg4[j] : 0.0;
              }
              if (last <= 1) trsm_update<1, false>(own, Lc, nr, kb, kw, row, col, acc);
              else if (last <= 2) trsm_update<2, false>(own, Lc, nr, kb, kw, row, col, acc);
              else trsm_update<4, false>(own, Lc, nr, kb, kw, row, col, acc);
#pragma unroll
              for (int j = 0; j < 4; ++j)
                if (tg4[j]) *tg4[j] = acc[j];
            }
            __syncwarp();
          }
        }
        Lc += 32LL * (nr - kb) - 16 * 33;                          // panel row t of column kb + 32
      }
    }
  }
}

// The same for a whole chunk of 32 columns by one CTA, the triangle shared by its warps 8 rows at a time: the rows
// below read L's digits once for 32 columns instead of once for 8 or 16, the first of them while one warp solves, and
// every step of the triangle has a barrier.  Same operations in the same order as trsm_team, so the same bits.
// The planner takes it for batches of large subdomains (rule and figures in sc_plan.cpp).  Where the triangles must not
// be divided by their diagonals it runs behind trsm_split_kernel and takes the launch over; on ordinary factors that
// launch is empty, 3 to 4 us of a small assembly's 75 to 110.  As part of trsm_split_kernel, inlined or out of line, it
// cost the teams up to 8 % at 5 digits.
template <int S>
struct ChunkShared {
  double X[32][33];                              // the solved block: [row][live column]
  double T[32 * 31 / 2];
  __align__(16) __nv_bfloat16 PX[S][32][kPad];   // its digit planes: [digit][live column][row]
  int emax[32];
};

template <int S>
__device__ __forceinline__ void trsm_chunk(const PlanPtrs &P, int task, const double *__restrict__ Lv, const double *__restrict__ invd,
                           const TrsmSplit &sp, double *__restrict__ Y, ChunkShared<S> &sm, bool unscaled) {
  const TrsmTask t = P.trsm_tasks[task];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int g = lane >> 2, tg = lane & 3;
  const int c_hi = t.c_lo + t.w;
  // the warp that solves: spread over the SM's sub-partitions across co-resident CTAs
  const int tri = (int)(((unsigned)task * 2654435761u) >> 30);
  int *colexp = sp.colexp + P.subs[t.sub].col_off;
  for (int li = 0; li < t.list_len; ++li) {
    const SnDev s = P.sns[P.trsm_list[t.list_off + li]];
    const int a = max(s.jlo, t.c_lo), w = min(s.jhi, c_hi) - a, ws = s.jhi - s.jlo;
    double *Ys = Y + s.y_off + (a - s.jlo);
    for (int e = tid; e < s.ns * w; e += kThreads) {
      const int r = e / w;
      Ys[(int64_t)r * ws + e - r * w] = 0.0;
    }
  }
  __syncthreads();
  for (int e = t.seed_lo + tid; e < t.seed_hi; e += kThreads) Y[P.seeds[e].y_off] = P.seeds[e].value;
  __syncthreads();

  for (int li = 0; li < t.list_len; ++li) {
    const SnDev s = P.sns[P.trsm_list[t.list_off + li]];
    const int a = max(s.jlo, t.c_lo), b = min(s.jhi, c_hi), ws = s.jhi - s.jlo, colsh = a - s.jlo;
    double *Ys = Y + s.y_off + colsh;
    const double *id = invd + s.lcp_off;
    const int64_t *rm = P.rmap + s.rmap_off;
    const int nr = s.ns + s.rs;
    const double *Lc = Lv + P.lcp[s.lcp_off];                // panel row t of column kb at Lc + t
    for (int kb = 0, blk = 0; kb < s.ns; Lc += 32LL * (nr - kb) - 16 * 33, kb += 32, ++blk) {
      const int kw = min(32, s.ns - kb), below = kb + kw, nb = nr - below;
      const int wk = min(b, P.cuts[s.cut_off + blk]) - a;
      if (wk <= 0) continue;
      const int64_t base = s.ld_off + (int64_t)blk * nr - 16LL * blk * (blk + 1);
      Fragments<S, false> fr;
      auto load_fr = [&](int r0) { fr.load(sp, base + r0 + g, r0 + g < nb, r0 + g + 8 < nb, tg); };
      const bool pre = warp != tri && kw > kDirect && 16 * warp < nb;
      if (pre) load_fr(16 * warp);
      for (int e = tid; e < kw * 32; e += kThreads) {
        const int q = e >> 5, c = e & 31;
        sm.X[q][c] = c < wk ? Ys[(int64_t)(kb + q) * ws + c] : 0.0;
      }
      const bool scaled = kw > kDirect && !unscaled;
#pragma unroll 4
      for (int p = warp; p < kw; p += kThreads / 32)
        if (lane > p && lane < kw) {
          const double l = Lc[kb + lane + p * (nr - kb - 1) - p * (p - 1) / 2];
          sm.T[tri_at(lane, p)] = scaled ? l * id[kb + p] : l;
        }
      __syncthreads();
      for (int p0 = 0; p0 < kw; p0 += 8) {
        const int pe = min(p0 + 8, kw);
        if (warp == tri && lane < wk) {
          double x[8];
#pragma unroll
          for (int i = 0; i < 8; ++i) x[i] = p0 + i < kw ? sm.X[p0 + i][lane] : 0.0;
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            if (p0 + i >= kw) break;                         // uniform
            if (!scaled) x[i] *= id[kb + p0 + i];
#pragma unroll
            for (int r = i + 1; r < 8; ++r)
              if (p0 + r < kw) x[r] = fma(-sm.T[tri_at(p0 + r, p0 + i)], x[i], x[r]);
          }
#pragma unroll
          for (int i = 0; i < 8; ++i)
            if (p0 + i < kw) sm.X[p0 + i][lane] = x[i];
        }
        __syncthreads();
        if (pe < kw) {                                       // then pe == p0 + 8
          if (lane < wk) {
            double x[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) x[i] = sm.X[p0 + i][lane];
            for (int r = pe + ((warp - tri) & 3); r < kw; r += kThreads / 32) {
              double xr = sm.X[r][lane];
#pragma unroll
              for (int i = 0; i < 8; ++i) xr = fma(-sm.T[tri_at(r, p0 + i)], x[i], xr);
              sm.X[r][lane] = xr;
            }
          }
          __syncthreads();
        }
      }
      if (warp == tri) {
        int em = 0;
        if (lane < wk)
          for (int q = 0; q < kw; ++q) {
            double v = sm.X[q][lane];
            if (scaled) sm.X[q][lane] = v = v * id[kb + q];
            Ys[(int64_t)(kb + q) * ws + lane] = v;
            em = max(em, biased_exponent(v));
          }
        sm.emax[lane] = em;
        if (lane < wk && em) atomicMax(colexp + a + lane, em);
      }
      __syncthreads();
      if (nb <= 0) continue;                                 // uniform
      if (kw <= kDirect) {
        // (row, live column) pairs numbered row by row and dealt to the threads in turn
        const int dp = kThreads / wk, dc = kThreads - dp * wk;
        int p = below + tid / wk, cl = tid - tid / wk * wk;
        while (p < nr) {
          double *tgt = (p < s.ns ? Ys + (int64_t)p * ws : Y + rm[p - s.ns] + colsh) + cl;
          double acc = *tgt;
          int o = p;
          for (int q = 0; q < kw; ++q) {
            acc = fma(-Lc[o], sm.X[q][cl], acc);
            o += nr - (kb + q) - 1;
          }
          *tgt = acc;
          p += dp;
          cl += dc;
          if (cl >= wk) {
            cl -= wk;
            ++p;
          }
        }
        __syncthreads();
        continue;
      }
      for (int e = tid; e < 32 * 32; e += kThreads) {
        const int q = e >> 5, c = e & 31;
        const double v = (q < kw && c < wk) ? sm.X[q][c] : 0.0;
        const uint64_t m = fixed_point(v, sm.emax[c]);
#pragma unroll
        for (int d = 0; d < S; ++d) sm.PX[d][c][q] = digit_bf16(m, d, v < 0.0);
      }
      __syncthreads();
      for (int r0 = 16 * warp; r0 < nb; r0 += 16 * (kThreads / 32)) {
        const int ra = r0 + g, rb = r0 + g + 8;
        const bool va = ra < nb, vb = rb < nb;
        const int ea = va ? sp.lexp[base + ra] : 0, eb = vb ? sp.lexp[base + rb] : 0;
        double *ta = nullptr, *tb = nullptr;                 // this lane's two target rows
        if (va) ta = Y + colsh + (below + ra < s.ns ? s.y_off + (int64_t)(below + ra) * ws : rm[below + ra - s.ns]);
        if (vb) tb = Y + colsh + (below + rb < s.ns ? s.y_off + (int64_t)(below + rb) * ws : rm[below + rb - s.ns]);
        if (!(pre && r0 == 16 * warp)) load_fr(r0);
#pragma unroll
        for (int nt = 0; nt < 4; ++nt) {
          if (8 * nt >= wk) break;                           // uniform
          // the targets' current values, loaded before the products so that
          // their latency overlaps the MMAs
          double yv[4];
#pragma unroll
          for (int r = 0; r < 4; ++r) {
            const int col = 8 * nt + 2 * tg + (r & 1);
            const double *p = (r & 2) ? tb : ta;
            yv[r] = (p && col < wk) ? p[col] : 0.0;
          }
          Groups<S> gr[4];
#pragma unroll
          for (int d = 0; d < S; ++d) {
            float c[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
            for (int q = 0; q <= d; ++q) {
              const __nv_bfloat16 *px = &sm.PX[d - q][8 * nt + g][2 * tg];
              fr.mma(c, q, px);
            }
#pragma unroll
            for (int r = 0; r < 4; ++r) gr[r].add(d, __float2int_rn(c[r]));
          }
#pragma unroll
          for (int r = 0; r < 4; ++r) {
            const int col = 8 * nt + 2 * tg + (r & 1);
            double *p = (r & 2) ? tb : ta;
            if (p && col < wk) {
              const int e = ((r & 2 ? eb : ea) - 1022) + (sm.emax[col] - 1022) + Groups<S>::kBlockShift;
              const double v = (double)gr[r].block_int();
              p[col] = (e >= -1022 && e <= 1023) ? fma(-v, pow2i(e), yv[r]) : yv[r] - ldexp(v, e);
            }
          }
        }
      }
      __syncthreads();
    }
  }
}

// Resident CTAs: with C = 2 three (168 registers, 8 bytes of spills at 7 digits and none below: 2.9 -> 2.3 ms on eight
// elasticity cubes at 7 digits), with C = 4 four (128 registers, 128 / 72 / 32 bytes of spills at 7 / 6 / 5 digits and still
// 6.6 -> 6.3 ms on 64 heat cubes at 7).
template <int C, int S>
__global__ void __launch_bounds__(kThreads, C >= 4 ? 4 : 3) trsm_split_kernel(const PlanPtrs P, const double *__restrict__ Lv,
                                                              const double *__restrict__ invd, const TrsmSplit sp,
                                                              double *__restrict__ Y) {
  extern __shared__ __align__(16) unsigned char team_smem[];
  constexpr int kParts = kChunk / (4 * C);
  if (*sp.unscaled) return;                                        // trsm_chunk_kernel takes the launch over
  trsm_team<C, S>(P, P.trsm_tasks[blockIdx.x / kParts], blockIdx.x % kParts, Lv, invd, sp, Y,
                  *reinterpret_cast<TeamShared<C, S> *>(team_smem), threadIdx.x >> 5, threadIdx.x & 31);
}

template <int S>
__global__ void __launch_bounds__(kThreads, S <= 4 ? 6 : S == 5 ? 5 : 4) trsm_chunk_kernel(const PlanPtrs P, const double *__restrict__ Lv,
                                                                 const double *__restrict__ invd, const TrsmSplit sp,
                                                                 double *__restrict__ Y, bool always) {
  __shared__ ChunkShared<S> sm;
  const bool unscaled = *sp.unscaled != 0;
  if (always || unscaled) trsm_chunk<S>(P, blockIdx.x, Lv, invd, sp, Y, sm, unscaled);
}

}  // namespace

#define SC_SPLIT_SWITCH(S_, CALL) \
  switch (S_) {                   \
    case 3: CALL(3); break;       \
    case 4: CALL(4); break;       \
    case 5: CALL(5); break;       \
    case 6: CALL(6); break;       \
    default: CALL(7); break;      \
  }

int launch_lpack_split(const sc_ctx &c, int S_, int64_t base, int64_t count, const double *Lv, void *ws,
                       void *stream) {
  if (count <= 0) return (int)cudaGetLastError();
  const cudaStream_t st = static_cast<cudaStream_t>(stream);
  uint8_t *w = static_cast<uint8_t *>(ws);
  __nv_bfloat16 *Ld = reinterpret_cast<__nv_bfloat16 *>(w + c.ws.ld_off);
  int16_t *lexp = reinterpret_cast<int16_t *>(w + c.ws.lexp_off);
  PlanPtrs p = c.ptrs();
  p.sblk += 2 * base;
#define LP(S) lpack_kernel<S><<<(unsigned)count, kThreads, 0, st>>>(p, Lv, Ld, lexp, c.ws.ld_rows)
  SC_SPLIT_SWITCH(S_, LP)
#undef LP
  return (int)cudaGetLastError();
}

template <int C, int S>
static void launch_team(const PlanPtrs &p, int n, const double *Lv, const double *invd, const TrsmSplit &sp, double *Y,
                        cudaStream_t st) {
  const int smem = (int)sizeof(TeamShared<C, S>);
  cudaFuncSetAttribute(trsm_split_kernel<C, S>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  trsm_split_kernel<C, S><<<(unsigned)(n * (kChunk / (4 * C))), kThreads, smem, st>>>(p, Lv, invd, sp, Y);
}

int launch_trsm_split(const sc_ctx &c, int S_, int cols, int64_t base, int64_t count, const double *Lv,
                      const double *invd, void *ws, double *Y, void *stream) {
  if (count <= 0) return (int)cudaGetLastError();
  const cudaStream_t st = static_cast<cudaStream_t>(stream);
  uint8_t *w = static_cast<uint8_t *>(ws);
  const TrsmSplit sp{reinterpret_cast<const __nv_bfloat16 *>(w + c.ws.ld_off),
                     reinterpret_cast<const int16_t *>(w + c.ws.lexp_off), c.ws.ld_rows,
                     reinterpret_cast<int *>(w + c.ws.colexp_off),
                     reinterpret_cast<const unsigned *>(w + c.ws.status_off) + kUnscaledWord};
  PlanPtrs p = c.ptrs();
  p.trsm_tasks += base;
#define TS(S)                                                                                                   \
  if (cols == 2) launch_team<2, S>(p, (int)count, Lv, invd, sp, Y, st);                                         \
  else if (cols == 4) launch_team<4, S>(p, (int)count, Lv, invd, sp, Y, st);                                    \
  trsm_chunk_kernel<S><<<(unsigned)count, kThreads, 0, st>>>(p, Lv, invd, sp, Y, cols >= 8)
  SC_SPLIT_SWITCH(S_, TS)
#undef TS
  return (int)cudaGetLastError();
}

int launch_yslice_group(const sc_ctx &c, int S_, int64_t base, int64_t count, const double *Y, void *ws,
                        void *stream, bool balanced) {
  if (count <= 0) return (int)cudaGetLastError();
  const cudaStream_t st = static_cast<cudaStream_t>(stream);
  uint8_t *w = static_cast<uint8_t *>(ws);
  const int *colexp = reinterpret_cast<const int *>(w + c.ws.colexp_off);
  __nv_bfloat16 *Yd = reinterpret_cast<__nv_bfloat16 *>(w + c.ws.yd_off);
  PlanPtrs p = c.ptrs();
  p.sblk += 2 * base;
#define YS(S) yslice_kernel<S, false><<<(unsigned)count, kThreads, 0, st>>>(p, Y, colexp, Yd, c.ws.yd_plane)
#define YB(S) yslice_kernel<S, true><<<(unsigned)count, kThreads, 0, st>>>(p, Y, colexp, Yd, c.ws.yd_plane)
  if (balanced) {
    SC_SPLIT_SWITCH(S_, YB)
  } else {
    SC_SPLIT_SWITCH(S_, YS)
  }
#undef YS
#undef YB
  return (int)cudaGetLastError();
}

int launch_syrk_split(const sc_ctx &c, int S_, int64_t base, int64_t count, void *ws, double *F, void *stream) {
  if (count <= 0) return (int)cudaGetLastError();
  const cudaStream_t st = static_cast<cudaStream_t>(stream);
  uint8_t *w = static_cast<uint8_t *>(ws);
  const int *colexp = reinterpret_cast<const int *>(w + c.ws.colexp_off);
  const __nv_bfloat16 *Yd = reinterpret_cast<const __nv_bfloat16 *>(w + c.ws.yd_off);
  PlanPtrs p = c.ptrs();
  p.syrk_tasks += base;
#define SY(S)                                                                                              \
  {                                                                                                        \
    const int smem = (int)(4 * sizeof(__nv_bfloat16) * S * 32 * kPad);                                     \
    cudaFuncSetAttribute(syrk_split_kernel<S>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);         \
    syrk_split_kernel<S><<<(unsigned)count, kThreads, smem, st>>>(p, Yd, c.ws.yd_plane, colexp, F);        \
  }
  SC_SPLIT_SWITCH(S_, SY)
#undef SY
  return (int)cudaGetLastError();
}

}  // namespace sc
