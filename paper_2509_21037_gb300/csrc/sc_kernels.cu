// sm_103a kernels of the Schur-complement assembly and application (FP64).
//
//   prep_kernel   -- reciprocal of L's diagonal for every column of an active
//                    supernode; a non-positive / non-finite pivot sets the
//                    NOT_SPD bit of the workspace status word (paper Sec. 3.1:
//                    the factor is copied in; here its CSC columns are read
//                    in place, because a fundamental supernode's CSC column is
//                    already a dense trapezoidal panel column).
//   trsm_kernel   -- Y = L^{-1} P B^T on a part of a 32-column chunk of the
//                    pivot-sorted columns (paper Sec. 3.2), one warp to a part:
//                    zero + seed the part's nonzero rows of Y, then for each
//                    supernode the part reaches (children first) a blocked
//                    forward substitution: 32x32 diagonal triangle, then the
//                    GEMM update of every panel row below it -- the rest of the
//                    diagonal block and the pruned rows, whose results land in
//                    the ancestors' Y blocks.
//   syrk_kernel   -- one 32x32 block of F = Y^T Y in pivot-sorted order
//                    (paper Sec. 3.3), summed over the supernodes active on
//                    both chunks; the epilogue writes it straight into the
//                    user's column order (the final back-permutation).
//   apply_kernel  -- q += scatter(F_i gather(lambda)) reading each stored
//                    lower tile once and using it for both triangles.
//   export_kernel -- tile-packed F_i -> dense full column-major matrix.
//
// FP64 on GB300 is a narrow pipe (about 1.2 TFLOP/s for the whole GPU), so
// these kernels are bound by FP64 issue; the work they do is what the plan's
// sparsity pattern leaves, and how it is shared out (the planner's rules for
// trsm_cols and syrk_ctas) keeps every SM busy: one warp's serial triangle overlaps
// the others' updates.
#include <cuda_runtime.h>

#include <algorithm>

#include <cstdint>

#include "sc_internal.h"

namespace sc {

// One launch for what the stages need beforehand (two launches cost a small batch
// 3 us of its 60).  CTAs below nprep: reciprocal diagonal.  The others, one per
// subdomain: zero the entries of F beyond m (rows >= m of the last tile row and
// columns >= m of the last diagonal tile).
__global__ void __launch_bounds__(256) prep_kernel(const int64_t *__restrict__ lcp, const int32_t *__restrict__ active,
                                                   int64_t nact, int nprep, const double *__restrict__ Lv,
                                                   double *__restrict__ invd, uint32_t *__restrict__ status,
                                                   const SubDev *__restrict__ subs, double *__restrict__ F) {
  if ((int)blockIdx.x < nprep) {
    for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < nact; k += (int64_t)nprep * blockDim.x) {
      const int32_t g = active[k];
      const double d = Lv[lcp[g]];
      if (!(d > 0.0) || !isfinite(d)) {
        atomicOr(status, kStatusNotSpd);
        invd[g] = 0.0;
      } else {
        invd[g] = 1.0 / d;
      }
    }
    return;
  }
  const SubDev sd = subs[blockIdx.x - nprep];
  if (sd.nt == 0) return;
  const int rem = sd.m - (sd.nt - 1) * kTile;
  if (rem == kTile) return;
  const int I = sd.nt - 1;
  double *T = F + sd.F_off + (int64_t)I * (I + 1) / 2 * (kTile * kTile);   // the last tile row, tile by tile
  const int total = (I + 1) * kTile * kTile;
  for (int e = threadIdx.x; e < total; e += blockDim.x) {
    const int r = e & (kTile - 1), c = e / kTile;         // c: column of the whole tile row
    if (r >= rem || c >= sd.m) T[e] = 0.0;
  }
}

// dst (shared) := src, or 0 where !in (src is then not read); 8-byte aligned
__device__ __forceinline__ void cp_async8(double *dst, const double *src, bool in) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;\n" ::"r"((uint32_t)__cvta_generic_to_shared(dst)),
               "l"(src), "r"(in ? 8 : 0)
               : "memory");
}

// ---- sparse TRSM ----------------------------------------------------------
//
// A warp solves the columns of one part of a 32-column chunk on its own: W
// columns, W a power of two, so that a chunk is 32 / W parts and no warp waits
// for another.  It walks the supernodes that its columns reach (children
// first); per 32-row block the triangle is solved with the block's rows of Y in
// registers, then every row below is updated.  A part of few columns reaches
// few supernodes, and a batch of few chunks still fills the GPU; the price
// is that L is read once per part and that a triangle uses fewer of the lanes.
// Every entry of Y is one chain of multiply-adds in column order, whatever W.
//
// Bound by FP64 issue on a large batch and by the longest part's chain on a small
// one.  Against one CTA of four warps per 32-column chunk (two to six barriers a
// block): one square 180 -> 32 us, 36 plane squares 1.01 -> 0.28 ms, eight
// elasticity cubes 20.0 -> 7.8 ms, 64 heat cubes 17.5 -> 17.4 ms (1.14 TFLOP/s of useful work).

constexpr int kTrsmCtas = 4;   // resident CTAs per SM: 128 registers a thread (at 96 and 80 they spill: 7.8 -> 8.8 ms on eight elasticity cubes)

// What a warp keeps of a listed supernode.
struct TrsmSn {
  int64_t y_off, rmap_off, lval;      // lval: index of L(c0, c0)
  int32_t ns, rs, jlo, jhi, cut_off, lcp_off;
};

template <int W>
struct TrsmShared {
  double X[32][W];            // the solved block: [row][live column]
  double T[32 * 31 / 2];      // the block's triangle below the diagonal, column by column
  TrsmSn sn[32];
};

// entry (row, p) of the packed triangle, row > p
__device__ __forceinline__ int tri_at(int row, int p) { return p * 31 - p * (p - 1) / 2 + row - p - 1; }

// The triangle of one block with V >= wk lanes across the live columns: lane
// = (row slot, column), NP pieces of 32 / V rows (NP a constant: a row update that
// is only predicated off would hold the FP64 pipe all the same).
template <int V, int NP, int W>
__device__ __forceinline__ void trsm_pieces(TrsmShared<W> &sm, double *__restrict__ Yb, int ws, int kw, int wk,
                                            double idv, int lane) {
  constexpr int RP = 32 / V;          // rows per piece
  const int cl = lane % V, rs = lane / V;
  double x[NP];
#pragma unroll
  for (int i = 0; i < NP; ++i) {
    const int r = i * RP + rs;
    x[i] = (r < kw && cl < wk) ? Yb[(int64_t)r * ws + cl] : 0.0;
  }
#pragma unroll
  for (int i = 0; i < NP; ++i) {
    const int k1 = min(RP, kw - i * RP);
#pragma unroll 2
    for (int k = 0; k < k1; ++k) {
      const int p = i * RP + k;
      const double xp = __shfl_sync(0xffffffffu, x[i], k * V + cl) * __shfl_sync(0xffffffffu, idv, p);
      if (rs == k) x[i] = xp;
#pragma unroll
      for (int j = i; j < NP; ++j) {
        const int r = j * RP + rs;
        if (r > p && r < kw) x[j] = fma(-sm.T[tri_at(r, p)], xp, x[j]);
      }
    }
  }
#pragma unroll
  for (int i = 0; i < NP; ++i) {
    const int r = i * RP + rs;
    if (r < kw && cl < wk) {
      Yb[(int64_t)r * ws + cl] = x[i];
      sm.X[r][cl] = x[i];
    }
  }
}

template <int V, int W>
__device__ __forceinline__ void trsm_triangle(TrsmShared<W> &sm, double *__restrict__ Yb, int ws, int kw, int wk,
                                              double idv, int lane) {
  if (V >= 2 && wk <= V / 2) {
    trsm_triangle<(V >= 2 ? V / 2 : 1), W>(sm, Yb, ws, kw, wk, idv, lane);
    return;
  }
  const int np = (kw + 32 / V - 1) / (32 / V);
  if (np <= 1) trsm_pieces<V, 1, W>(sm, Yb, ws, kw, wk, idv, lane);
  else if (V >= 2 && np <= 2) trsm_pieces<V, (V >= 2 ? 2 : 1), W>(sm, Yb, ws, kw, wk, idv, lane);
  else if (V >= 4 && np <= 4) trsm_pieces<V, (V >= 4 ? 4 : 1), W>(sm, Yb, ws, kw, wk, idv, lane);
  else if (V >= 8 && np <= 8) trsm_pieces<V, (V >= 8 ? 8 : 1), W>(sm, Yb, ws, kw, wk, idv, lane);
  else trsm_pieces<V, V, W>(sm, Yb, ws, kw, wk, idv, lane);
}

// NJ (row, column) pairs per lane of the update below a block: acc -= L(row, block) X(:, column).
// kFlat: the pairs' columns differ; else they are all col[0].
template <int NJ, bool kFlat, int W>
__device__ __forceinline__ void trsm_update(const TrsmShared<W> &sm, const double *__restrict__ Lb, int nr, int kb,
                                            int kw, const int (&row)[4], const int (&col)[4], double (&acc)[4]) {
  const double *lp[NJ];
#pragma unroll
  for (int j = 0; j < NJ; ++j) lp[j] = Lb + row[j];
  int o = 0;
#pragma unroll 4
  for (int q = 0; q < kw; ++q) {
    const double x0 = sm.X[q][col[0]];
#pragma unroll
    for (int j = 0; j < NJ; ++j) acc[j] = fma(-lp[j][o], kFlat ? sm.X[q][col[j]] : x0, acc[j]);
    o += nr - (kb + q) - 1;           // from entry (row, c) of the panel to entry (row, c + 1)
  }
}

template <int W>
__device__ __forceinline__ void trsm_part(const PlanPtrs &P, const TrsmTask &t, int part,
                                          const double *__restrict__ Lv, const double *__restrict__ invd,
                                          double *__restrict__ Y, TrsmShared<W> &sm, int lane) {
  const int c_lo = t.c_lo + part * W, c_hi = min(c_lo + W, t.c_lo + t.w);
  if (c_lo >= c_hi) return;

  // the next 32 listed supernodes, those that the part reaches into sm.sn
  auto batch = [&](int l0) -> int {
    bool hit = false;
    SnDev s{};
    if (l0 + lane < t.list_len) {
      s = P.sns[P.trsm_list[t.list_off + l0 + lane]];
      hit = max(s.jlo, c_lo) < min(s.jhi, c_hi);
    }
    const uint32_t m = __ballot_sync(0xffffffffu, hit);
    __syncwarp();
    if (hit) {
      TrsmSn &e = sm.sn[__popc(m & ((1u << lane) - 1))];
      e.y_off = s.y_off; e.rmap_off = s.rmap_off; e.lval = P.lcp[s.lcp_off];
      e.ns = s.ns; e.rs = s.rs; e.jlo = s.jlo; e.jhi = s.jhi; e.cut_off = s.cut_off; e.lcp_off = s.lcp_off;
    }
    __syncwarp();
    return __popc(m);
  };

  // zero the part's columns of every Y block it reaches, then its entries of B^T
  int n = 0;
  for (int l0 = 0; l0 < t.list_len; l0 += 32) {
    n = batch(l0);
    for (int i = 0; i < n; ++i) {
      const TrsmSn &s = sm.sn[i];
      const int j = c_lo + lane % W, ws = s.jhi - s.jlo;
      if (j >= s.jlo && j < min(s.jhi, c_hi))
        for (int r = lane / W; r < s.ns; r += 32 / W) Y[s.y_off + (int64_t)r * ws + j - s.jlo] = 0.0;
    }
  }
  __syncwarp();
  {
    const int32_t *sp = P.seed_ptr + P.subs[t.sub].col_off;
    const int e1 = sp[c_hi];
    for (int e = sp[c_lo] + lane; e < e1; e += 32) Y[P.seeds[e].y_off] = P.seeds[e].value;
  }
  __syncwarp();

  for (int l0 = 0; l0 < t.list_len; l0 += 32) {
    if (t.list_len > 32) n = batch(l0);      // else it is there from the first walk
    for (int i = 0; i < n; ++i) {
      const TrsmSn s = sm.sn[i];
      const int a = max(s.jlo, c_lo), b = min(s.jhi, c_hi), ws = s.jhi - s.jlo, colsh = a - s.jlo;
      double *Ys = Y + s.y_off + colsh;
      const int64_t *rm = P.rmap + s.rmap_off;
      const int nr = s.ns + s.rs;
      // Lc[t]: panel row t of column kb (rows above the diagonal excepted)
      const double *Lc = Lv + s.lval;
      for (int kb = 0; kb < s.ns; kb += 32) {
        const int kw = min(32, s.ns - kb);
        // columns at or after the block's cut are still zero in these rows
        const int wk = min(b, P.cuts[s.cut_off + (kb >> 5)]) - a;
        if (wk > 0) {
          const double idv = lane < kw ? invd[s.lcp_off + kb + lane] : 0.0;
          {
            const double *lp = Lc + kb + lane;
            for (int p = 0; p < kw; ++p) {
              if (lane > p && lane < kw) cp_async8(&sm.T[tri_at(lane, p)], lp, true);
              lp += nr - (kb + p) - 1;
            }
            asm volatile("cp.async.commit_group;\n" ::: "memory");
          }
          // The (row, live column) pairs below the block, four to a lane at a time.  kFlat numbers
          // them row by row, so that every lane works whatever wk is; else lanes
          // past the last whole row idle and a lane keeps its column, whose X is then
          // loaded once (W = 16 on the 64-cube batch 17.67 -> 17.40 ms flat; W = 2 on eight
          // elasticity cubes 7.78 -> 8.81 ms, so not there).
          // The first pairs' targets do not depend on the triangle and are loaded before it.
          constexpr bool kFlat = W >= 16;
          const int below = kb + kw, dp = 32 / wk, dc = 32 - dp * wk;
          int p = below + lane / wk, cl = lane - lane / wk * wk;      // the lane's next pair
          if (!kFlat && lane >= dp * wk) p = nr;
          int row[4], col[4];
          double *tg[4];
          double acc[4];
          auto targets = [&]() {
#pragma unroll
            for (int j = 0; j < 4; ++j) {
              const bool ok = p < nr;
              row[j] = ok ? p : nr - 1;
              col[j] = cl;
              tg[j] = !ok ? nullptr : p < s.ns ? Ys + (int64_t)p * ws + cl : Y + rm[p - s.ns] + colsh + cl;
              acc[j] = ok ? *tg[j] : 0.0;
              p += dp;
              if (kFlat) {
                cl += dc;
                if (cl >= wk) {
                  cl -= wk;
                  ++p;
                }
              }
            }
          };
          int left = kFlat ? ((nr - below) * wk + 31) >> 5 : (nr - below + dp - 1) / dp;   // warp steps to do
          if (left > 0) targets();
          asm volatile("cp.async.wait_group 0;\n" ::: "memory");
          __syncwarp();
          double *Yb = Ys + (int64_t)kb * ws;
          trsm_triangle<W, W>(sm, Yb, ws, kw, wk, idv, lane);
          __syncwarp();
          while (left > 0) {
            switch (min(4, left)) {
              case 1: trsm_update<1, kFlat, W>(sm, Lc, nr, kb, kw, row, col, acc); break;
              case 2: trsm_update<2, kFlat, W>(sm, Lc, nr, kb, kw, row, col, acc); break;
              case 3: trsm_update<3, kFlat, W>(sm, Lc, nr, kb, kw, row, col, acc); break;
              default: trsm_update<4, kFlat, W>(sm, Lc, nr, kb, kw, row, col, acc); break;
            }
#pragma unroll
            for (int j = 0; j < 4; ++j)
              if (tg[j]) *tg[j] = acc[j];
            left -= 4;
            if (left > 0) targets();
          }
          __syncwarp();
        }
        // to column kb + 32: sum over the 32 columns of nr - c - 1
        Lc += 32LL * (nr - kb) - 16 * 33;
      }
    }
  }
}

// Work-queue form (queue != nullptr): a grid sized to the resident CTAs pulls
// parts from an atomic counter, a warp at a time; otherwise one CTA per four
// parts.  Tasks are ordered largest first by the planner.
template <int W>
__global__ void __launch_bounds__(kThreads, kTrsmCtas) trsm_kernel(const PlanPtrs P, const double *__restrict__ Lv,
                                                            const double *__restrict__ invd, double *__restrict__ Y,
                                                            unsigned *queue, int ntask) {
  constexpr int kParts = kChunk / W;
  __shared__ __align__(16) TrsmShared<W> smem[kThreads / 32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  TrsmShared<W> &sm = smem[warp];
  if (!queue) {
    const int k = (int)blockIdx.x * (kThreads / 32) + warp;
    if (k < ntask * kParts) trsm_part<W>(P, P.trsm_tasks[k / kParts], k % kParts, Lv, invd, Y, sm, lane);
    return;
  }
  for (;;) {
    int k = 0;
    if (lane == 0) k = (int)atomicAdd(queue, 1u);
    k = __shfl_sync(0xffffffffu, k, 0);
    if (k >= ntask * kParts) break;
    trsm_part<W>(P, P.trsm_tasks[k / kParts], k % kParts, Lv, invd, Y, sm, lane);
  }
}

// A 32x32 block of F (sorted chunks q1 >= q2) is cut into pieces of 8 rows and
// 4 NC columns; a lane holds row lane >> 2 and columns NC (lane & 3) .. of a
// piece.  With NP = 4 and NC = 2 one CTA does the block: warp w of an
// off-diagonal block takes a quadrant, the ten lower pieces of a diagonal block
// are dealt 3, 3, 2, 2.  With NP = 1 every warp has one piece and the block is
// shared by 4 (NC = 2) or 8 (NC = 1) CTAs: a row then holds a warp for two FP64
// instructions or one instead of eight.
template <int NP, int NC>
struct SyrkPieces {
  static constexpr int kCtas = NP > 1 ? 1 : 8 / NC;
  int n, rb[NP], cb[NP];
  __device__ __forceinline__ SyrkPieces(bool diag, int part, int w) {
    if constexpr (NP > 1) {
      // (row, column) of a diagonal block's pieces, two bits each, first piece lowest
      const uint32_t code = w == 0 ? 0x073u : w == 1 ? 0x1fbu : w == 2 ? 0x062u : 0x05au;
      n = !diag ? 4 : w < 2 ? 3 : 2;
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        rb[i] = diag ? (int)(code >> (4 * i)) & 3 : 2 * (w >> 1) + (i >> 1);
        cb[i] = diag ? (int)(code >> (4 * i + 2)) & 3 : 2 * (w & 1) + (i & 1);
      }
    } else {
      constexpr int kCols = 8 / NC;                    // pieces across a block
      const int u = part * (kThreads / 32) + w;
      n = 1;
      rb[0] = u / kCols;
      cb[0] = u % kCols;
      if (diag) {                                      // row r of pieces has the first (r + 1) kCols / 4
        int r = 0;
        while (r < 4 && u >= (r + 1) * (r + 2) / 2 * (kCols / 4)) ++r;
        n = r < 4 ? 1 : 0;
        rb[0] = r & 3;
        cb[0] = n ? u - r * (r + 1) / 2 * (kCols / 4) : 0;
      }
    }
  }
};

constexpr int kSyrkBatch = 64;   // supernodes whose rows are numbered through at a time

struct SyrkShared {
  double A[2][32][32], B[2][32][32];   // [stage][row of Y][column of chunk q1 / q2]
  int64_t off[kSyrkBatch];             // Y offset of (first live row, sorted column 0)
  int start[kSyrkBatch + 1];           // first row number of every supernode of the batch
  int ws[kSyrkBatch], jlo[kSyrkBatch], jhi[kSyrkBatch], cut[kSyrkBatch];
  int wsum, next;
};

// One SYRK task.  The rows of Y that are live on both chunks (of every listed
// supernode the rows from its first 32-row block whose cut lies beyond q1's
// first column) are numbered through and taken 32 at a time, whatever
// supernode they belong to: a plane domain's lists are mostly supernodes of one
// to three columns.  The next 32 rows are copied asynchronously while
// these are multiplied; a piece skips the rows on which its 8 rows or its 8
// columns are zero.  Every entry of F is one chain of multiply-adds in list order.
// Bound by FP64 issue (99 % of the pipe on eight heat cubes): what counts is the number of warp
// multiply-adds, a predicated one included.  Against one stage per supernode block and 32x32 blocks
// without pieces: 64 heat cubes 31.42 -> 30.26 ms (4 % fewer multiply-adds; 1.23 TFLOP/s of useful
// work), eight elasticity cubes 6.68 -> 6.46 ms, 36 plane squares 355 -> 153 us, one square 82 -> 14 us.
template <int NP, int NC>
__device__ __forceinline__ void syrk_task(const PlanPtrs &P, const SyrkTask t, int part, const double *__restrict__ Y,
                                          double *__restrict__ F, SyrkShared &sm, int rot) {
  const SubDev sd = P.subs[t.sub];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const bool diag = t.q1 == t.q2;
  const int j1lo = t.q1 * kChunk, j2lo = t.q2 * kChunk;
  const SyrkPieces<NP, NC> pc(diag, part, (warp + rot) & 3);
  if (diag && SyrkPieces<NP, NC>(true, part, 0).n == 0) return;   // no piece for this CTA (uniform)
  const int lr = lane >> 2, lc = NC * (lane & 3);
  double acc[NP][NC];
#pragma unroll
  for (int i = 0; i < NP; ++i)
#pragma unroll
    for (int h = 0; h < NC; ++h) acc[i][h] = 0.0;

  for (int l0 = 0; l0 < t.list_len; l0 += kSyrkBatch) {
    int n = 0;
    if (tid < kSyrkBatch && l0 + tid < t.list_len) {
      const SnDev s = P.sns[P.syrk_list[t.list_off + l0 + tid]];
      const int nb = (s.ns + 31) >> 5;
      int b = 0;
      while (b < nb && P.cuts[s.cut_off + b] <= j1lo) ++b;   // the cuts of a supernode do not decrease
      n = max(0, s.ns - 32 * b);
      const int ws = s.jhi - s.jlo;
      sm.off[tid] = s.y_off + (int64_t)(32 * b) * ws - s.jlo;
      sm.ws[tid] = ws;
      sm.jlo[tid] = s.jlo;
      sm.jhi[tid] = s.jhi;
      sm.cut[tid] = s.cut_off + b;
    }
    int inc = n;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const int v = __shfl_up_sync(0xffffffffu, inc, d);
      if (lane >= d) inc += v;
    }
    if (tid == 31) sm.wsum = inc;
    __syncthreads();
    if (tid < kSyrkBatch) sm.start[tid + 1] = inc + (warp == 1 ? sm.wsum : 0);
    if (tid == 0) sm.start[0] = 0;
    __syncthreads();
    const int total = sm.start[kSyrkBatch];

    // copies rows 32 st .. + 31 into stage st & 1; bit i of the result says
    // whether row 32 st + lane is live on this warp's piece i
    auto fetch = [&](int st) -> uint32_t {
      const int g = 32 * st + lane;
      int64_t off = 0;
      uint32_t rng = 0, need = 0;
      if (g < total) {
        int e = 0;
#pragma unroll
        for (int h = kSyrkBatch / 2; h >= 1; h >>= 1)
          if (sm.start[e + h] <= g) e += h;      // the last supernode that starts at or before row g
        const int r = g - sm.start[e];
        off = sm.off[e] + (int64_t)r * sm.ws[e];
        const int hi = min(sm.jhi[e], P.cuts[sm.cut[e] + (r >> 5)]), lo = sm.jlo[e];
        const int a1 = max(lo - j1lo, 0), b1 = min(hi - j1lo, 32), a2 = max(lo - j2lo, 0), b2 = min(hi - j2lo, 32);
        rng = (uint32_t)(a1 | b1 << 8 | a2 << 16 | b2 << 24);
#pragma unroll
        for (int i = 0; i < NP; ++i) {
          const int r0 = 8 * pc.rb[i], c0 = 4 * NC * pc.cb[i];
          if (i < pc.n && a1 < r0 + 8 && b1 > r0 && a2 < c0 + 4 * NC && b2 > c0) need |= 1u << i;
        }
      }
      double(*As)[32] = sm.A[st & 1], (*Bs)[32] = sm.B[st & 1];
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const int k = 8 * warp + i;
        const int64_t o = __shfl_sync(0xffffffffu, off, k);
        const uint32_t q = __shfl_sync(0xffffffffu, rng, k);
        const bool ina = lane >= (int)(q & 0xff) && lane < (int)(q >> 8 & 0xff);
        const bool inb = lane >= (int)(q >> 16 & 0xff) && lane < (int)(q >> 24);
        cp_async8(&As[k][lane], ina ? Y + o + j1lo + lane : Y, ina);
        if (!diag) cp_async8(&Bs[k][lane], inb ? Y + o + j2lo + lane : Y, inb);
      }
      asm volatile("cp.async.commit_group;\n" ::: "memory");
      return need;
    };

    const int nst = (total + 31) >> 5;
    uint32_t need = nst > 0 ? fetch(0) : 0u;
    for (int st = 0; st < nst; ++st) {
      uint32_t nneed = 0;
      if (st + 1 < nst) {
        nneed = fetch(st + 1);
        asm volatile("cp.async.wait_group 1;\n" ::: "memory");
      } else {
        asm volatile("cp.async.wait_group 0;\n" ::: "memory");
      }
      __syncthreads();
      const double(*As)[32] = sm.A[st & 1], (*Bs)[32] = diag ? sm.A[st & 1] : sm.B[st & 1];
      const int kk = min(32, total - 32 * st);
      auto row = [&](int k, int i) {
        const double a = As[k][8 * pc.rb[i] + lr];
        const double *bp = &Bs[k][4 * NC * pc.cb[i] + lc];
        if constexpr (NC == 2) {
          const double2 b = *reinterpret_cast<const double2 *>(bp);
          acc[i][0] = fma(a, b.x, acc[i][0]);
          acc[i][1] = fma(a, b.y, acc[i][1]);
        } else {
          acc[i][0] = fma(a, *bp, acc[i][0]);
        }
      };
      // runs of rows with the same live pieces (a supernode's rows, mostly); a piece's rows are a
      // loop of their own, since a predicated multiply-add would hold the FP64 pipe all the same
      for (int k = 0; k < kk;) {
        const uint32_t m = __shfl_sync(0xffffffffu, need, k);
        const uint32_t other = __ballot_sync(0xffffffffu, need != m || lane >= kk) >> k;
        const int k1 = other ? k + __ffs(other) - 1 : 32;
        if (m == (1u << NP) - 1) {
#pragma unroll 4
          for (int q = k; q < k1; ++q)
#pragma unroll
            for (int i = 0; i < NP; ++i) row(q, i);
        } else {
#pragma unroll
          for (int i = 0; i < NP; ++i)
            if (m >> i & 1) {
#pragma unroll 4
              for (int q = k; q < k1; ++q) row(q, i);
            }
        }
        k = k1;
      }
      __syncthreads();               // the next copies overwrite this stage (or the next batch the tables)
      need = nneed;
    }
  }
  const int32_t *perm = P.perm_cols + sd.col_off;
#pragma unroll
  for (int i = 0; i < NP; ++i) {
    if (i >= pc.n) continue;
#pragma unroll
    for (int h = 0; h < NC; ++h) {
      const int r = 8 * pc.rb[i] + lr, c = 4 * NC * pc.cb[i] + lc + h;
      const int j1 = j1lo + r, j2 = j2lo + c;
      if (j1 < sd.m && j2 < sd.m && (!diag || r >= c)) {
        const int a = perm[j1], b = perm[j2];
        const int hi = max(a, b), lo = min(a, b);
        const int I = hi / kTile, J = lo / kTile;
        double *T = F + sd.F_off + ((int64_t)I * (I + 1) / 2 + J) * (kTile * kTile);
        T[(hi % kTile) + kTile * (lo % kTile)] = acc[i][h];
        if (I == J) T[(lo % kTile) + kTile * (hi % kTile)] = acc[i][h];
      }
    }
  }
}

// A rotation of a CTA's warps over its shares: a CTA's warps sit on the SM's four sub-partitions, so that
// equal shares on equal warps would load one FP64 pipe more than the others.
__device__ __forceinline__ int spread(unsigned k) { return (int)((k * 2654435761u) >> 30); }

template <int NP, int NC>
__global__ void __launch_bounds__(kThreads, 6) syrk_kernel(const PlanPtrs P, const double *__restrict__ Y,
                                                           double *__restrict__ F, unsigned *queue, int ntask) {
  constexpr int kCtas = SyrkPieces<NP, NC>::kCtas;
  __shared__ __align__(16) SyrkShared sm;
  if (!queue) {
    syrk_task<NP, NC>(P, P.syrk_tasks[blockIdx.x / kCtas], blockIdx.x % kCtas, Y, F, sm, spread(blockIdx.x));
    return;
  }
  for (;;) {
    if (threadIdx.x == 0) sm.next = (int)atomicAdd(queue, 1u);
    __syncthreads();
    const int k = sm.next;
    __syncthreads();
    if (k >= ntask * kCtas) break;
    syrk_task<NP, NC>(P, P.syrk_tasks[k / kCtas], k % kCtas, Y, F, sm, spread((unsigned)k));
    __syncthreads();
  }
}

__global__ void __launch_bounds__(kThreads) apply_kernel(const PlanPtrs P, const double *__restrict__ F,
                                                         const double *__restrict__ lam,
                                                         double *__restrict__ q) {
  __shared__ double Ts[kThreads / 32][32][33];
  __shared__ double red[kThreads / 32][32];
  const ApplyTask t = P.apply_tasks[blockIdx.x];
  const SubDev sd = P.subs[t.sub];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int32_t *map = P.lambda + sd.col_off;
  const int I = t.I;
  const int rowI = I * kTile + lane;
  const double pI = rowI < sd.m ? lam[map[rowI]] : 0.0;
  double y = 0.0;
  for (int J = warp; J <= I; J += kThreads / 32) {
    const double *Tg = F + sd.F_off + ((int64_t)I * (I + 1) / 2 + J) * (kTile * kTile);
#pragma unroll 8
    for (int c = 0; c < 32; ++c) Ts[warp][c][lane] = Tg[c * 32 + lane];
    __syncwarp();
    const int colJ = J * kTile + lane;
    const double pJ = colJ < sd.m ? lam[map[colJ]] : 0.0;
#pragma unroll 8
    for (int c = 0; c < 32; ++c) y = fma(Ts[warp][c][lane], __shfl_sync(0xffffffffu, pJ, c), y);
    if (J < I) {
      double z = 0.0;
#pragma unroll 8
      for (int r = 0; r < 32; ++r) z = fma(Ts[warp][lane][r], __shfl_sync(0xffffffffu, pI, r), z);
      if (colJ < sd.m) atomicAdd(q + map[colJ], z);
    }
    __syncwarp();
  }
  red[warp][lane] = y;
  __syncthreads();
  if (warp == 0) {
    double s = 0.0;
#pragma unroll
    for (int w = 0; w < kThreads / 32; ++w) s += red[w][lane];
    if (rowI < sd.m) atomicAdd(q + map[rowI], s);
  }
}

__global__ void export_kernel(const SubDev *__restrict__ subs, int32_t i, const double *__restrict__ F,
                              double *__restrict__ dst, int32_t ld) {
  const SubDev sd = subs[i];
  const int64_t total = (int64_t)sd.m * sd.m;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int a = (int)(e % sd.m), b = (int)(e / sd.m);
    const int hi = max(a, b), lo = min(a, b);
    const int I = hi / kTile, J = lo / kTile;
    const double *T = F + sd.F_off + ((int64_t)I * (I + 1) / 2 + J) * (kTile * kTile);
    dst[a + (int64_t)b * ld] = T[(hi % kTile) + kTile * (lo % kTile)];
  }
}

// ---------------------------------------------------------------------------
// launchers

static inline cudaStream_t S(void *s) { return static_cast<cudaStream_t>(s); }

// CTAs of `kernel` (kThreads threads, static shared memory) the GPU keeps resident at once
template <class K>
int resident_ctas(K kernel) {
  int dev = 0, sms = 0, per = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kernel, kThreads, 0);
  return std::max(1, sms * std::max(1, per));
}

int launch_prep(const sc_ctx &c, const double *Lv, double *invd, uint32_t *status, double *F, void *ws,
                void *stream) {
  const PlanPtrs p = c.ptrs();
  const int nprep = (int)std::min<int64_t>((c.n_active_cols + 255) / 256, 152 * 16);
  if (nprep + c.nsub > 0)
    prep_kernel<<<(unsigned)(nprep + c.nsub), 256, 0, S(stream)>>>(p.lcp, p.active_cols, c.n_active_cols, nprep, Lv,
                                                                   invd, status, p.subs, F);
  int e = (int)cudaGetLastError();
  if (!e && c.n_slices > 0) e = launch_colexp_reset(c, ws, stream);
  return e;
}

template <int W>
void launch_trsm(const sc_ctx &c, const PlanPtrs &p, int n, const double *Lv, const double *invd, void *ws, double *Y,
                 void *stream) {
  const int parts = n * (kChunk / W), ctas = (parts + kThreads / 32 - 1) / (kThreads / 32);
  cudaFuncSetAttribute(trsm_kernel<W>, cudaFuncAttributePreferredSharedMemoryCarveout,
                       (int)(kTrsmCtas * (sizeof(TrsmShared<W>) * 4 + 1024) * 100 / (228 * 1024)) + 1);
  if (c.persistent) {
    unsigned *q = reinterpret_cast<unsigned *>(static_cast<uint8_t *>(ws) + c.ws.status_off + 64);
    if (cudaMemsetAsync(q, 0, sizeof(unsigned), S(stream)) != cudaSuccess) return;   // the caller reads the error
    const int grid = std::min(ctas, resident_ctas(trsm_kernel<W>));
    trsm_kernel<W><<<(unsigned)grid, kThreads, 0, S(stream)>>>(p, Lv, invd, Y, q, n);
  } else {
    trsm_kernel<W><<<(unsigned)ctas, kThreads, 0, S(stream)>>>(p, Lv, invd, Y, nullptr, n);
  }
}

// First half of one variant group's pipeline: (digit planes of L,) sparse TRSM.
int launch_group_trsm(const sc_ctx &c, int w, int v, const double *Lv, const double *invd, void *ws, double *Y,
                      void *stream) {
  const auto &G = c.waves[w];
  if (v == 0) {
    if (G.trsm[0][1] > 0) {
      PlanPtrs p = c.ptrs();
      p.trsm_tasks += G.trsm[0][0];
      const int n = (int)G.trsm[0][1];
      switch (G.trsm_cols) {
        case 1: launch_trsm<1>(c, p, n, Lv, invd, ws, Y, stream); break;
        case 2: launch_trsm<2>(c, p, n, Lv, invd, ws, Y, stream); break;
        case 4: launch_trsm<4>(c, p, n, Lv, invd, ws, Y, stream); break;
        case 8: launch_trsm<8>(c, p, n, Lv, invd, ws, Y, stream); break;
        default: launch_trsm<16>(c, p, n, Lv, invd, ws, Y, stream); break;
      }
    }
    return (int)cudaGetLastError();
  }
  const int S = var_digits(v);
  int e = launch_lpack_split(c, S, G.sblk[v][0], G.sblk[v][1], Lv, ws, stream);
  if (!e) e = launch_trsm_split(c, S, G.trsm[v][0], G.trsm[v][1], Lv, invd, ws, Y, stream);
  return e;
}

template <int NP, int NC>
void launch_syrk(const sc_ctx &c, const PlanPtrs &p, int n, const double *Y, void *ws, double *F, void *stream) {
  const int ctas = n * SyrkPieces<NP, NC>::kCtas;
  // six CTAs of 34 KB to an SM
  cudaFuncSetAttribute(syrk_kernel<NP, NC>, cudaFuncAttributePreferredSharedMemoryCarveout,
                       cudaSharedmemCarveoutMaxShared);
  if (c.persistent) {
    unsigned *q = reinterpret_cast<unsigned *>(static_cast<uint8_t *>(ws) + c.ws.status_off + 128);
    if (cudaMemsetAsync(q, 0, sizeof(unsigned), S(stream)) != cudaSuccess) return;   // the caller reads the error
    const int grid = std::min(ctas, resident_ctas(syrk_kernel<NP, NC>));
    syrk_kernel<NP, NC><<<(unsigned)grid, kThreads, 0, S(stream)>>>(p, Y, F, q, n);
  } else {
    syrk_kernel<NP, NC><<<(unsigned)ctas, kThreads, 0, S(stream)>>>(p, Y, F, nullptr, n);
  }
}

// Second half: (digit planes of Y,) pruned SYRK with the back permutation.
int launch_group_syrk(const sc_ctx &c, int w, int v, const double *Y, void *ws, double *F, void *stream) {
  const auto &G = c.waves[w];
  if (v == 0) {
    if (G.syrk[0][1] > 0) {
      PlanPtrs p = c.ptrs();
      p.syrk_tasks += G.syrk[0][0];
      const int n = (int)G.syrk[0][1];
      if (G.syrk_ctas == 8) launch_syrk<1, 1>(c, p, n, Y, ws, F, stream);
      else if (G.syrk_ctas == 4) launch_syrk<1, 2>(c, p, n, Y, ws, F, stream);
      else launch_syrk<4, 2>(c, p, n, Y, ws, F, stream);
    }
    return (int)cudaGetLastError();
  }
  const int S = var_digits(v);
  int e = launch_yslice_group(c, S, G.sblk[v][0], G.sblk[v][1], Y, ws, stream, (v & kVarTile) != 0);
  if (e) return e;
  if (v & kVarTile) return launch_syrk_tc(c, S, G.syrk[v][0], G.syrk[v][1], ws, F, stream);
  return launch_syrk_split(c, S, G.syrk[v][0], G.syrk[v][1], ws, F, stream);
}

int launch_apply(const sc_ctx &c, const double *F, const double *lam, double *q, void *stream) {
  if (c.n_apply > 0) apply_kernel<<<(unsigned)c.n_apply, kThreads, 0, S(stream)>>>(c.ptrs(), F, lam, q);
  return (int)cudaGetLastError();
}

int launch_export(const sc_ctx &c, const double *F, int32_t i, double *dst, int32_t ld, void *stream) {
  const int64_t total = (int64_t)c.m[i] * c.m[i];
  if (total > 0) {
    int64_t blocks = (total + 255) / 256;
    if (blocks > 152 * 16) blocks = 152 * 16;
    export_kernel<<<(unsigned)blocks, 256, 0, S(stream)>>>(c.ptrs().subs, i, F, dst, ld);
  }
  return (int)cudaGetLastError();
}

}  // namespace sc
