// The sparse TRSM of one part of a 32-column chunk by one warp in FP64 (sc_kernels.cu), and its pieces for the
// split-precision form (sc_split.cu).
#pragma once

#include <cstdint>

#include "sc_internal.h"

namespace sc {

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

// Split precision: blocks of at most kDirect columns update the rows below in FP64, a multiply-add per
// column and entry of Y against the two operations that an entry costs after the digit products.
constexpr int kDirect = 4;

// Resident CTAs per SM: 128 registers a thread, with which W = 16 spills 84 bytes and the others none; at 96 and 80 all do
// (7.8 -> 8.8 ms on eight elasticity cubes).
constexpr int kTrsmCtas = 4;

// What a warp keeps of a listed supernode.
struct TrsmSn {
  int64_t y_off, rmap_off, ld_off, lval;   // lval: index of L(c0, c0)
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
// is only predicated off would hold the FP64 pipe all the same).  kScaled: T holds L(row, p) / L(p, p), so that
// the chain is one multiply-add a step and the rows are divided at the end.  Every entry of L is rounded once more, so
// only the split-precision form does it, where that is lost in the digits' error (7 digits against 64 bits, six
// subdomains of cubes, squares and elasticity: 1.6e-15 to 6.8e-15 with it and without it; on the mean 0.98 and 0.97 of
// the error before), and only where FP64 holds the ratios in full (prep_kernel).  Without it, TRSM at 7 and 5 digits:
// 64 heat cubes 6.4 -> 6.6 and 5.0 -> 5.4 ms, four elasticity cubes 1.43 -> 1.47 and 1.18 -> 1.34.
template <int V, int NP, bool kScaled, class Sm>
__device__ __forceinline__ void trsm_pieces(Sm &sm, const double *__restrict__ T, double *__restrict__ Yb, int ws, int kw, int wk,
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
      double xp = __shfl_sync(0xffffffffu, x[i], k * V + cl);
      if (!kScaled) {
        xp *= __shfl_sync(0xffffffffu, idv, p);
        if (rs == k) x[i] = xp;
      }
#pragma unroll
      for (int j = i; j < NP; ++j) {
        const int r = j * RP + rs;
        if (r > p && r < kw) x[j] = fma(-T[tri_at(r, p)], xp, x[j]);
      }
    }
  }
#pragma unroll
  for (int i = 0; i < NP; ++i) {
    const int r = i * RP + rs;
    if (kScaled) x[i] *= __shfl_sync(0xffffffffu, idv, r & 31);
    if (r < kw && cl < wk) {
      Yb[(int64_t)r * ws + cl] = x[i];
      sm.X[r][cl] = x[i];
    }
  }
}

template <int V, bool kScaled, class Sm>
__device__ __forceinline__ void trsm_triangle(Sm &sm, const double *__restrict__ T, double *__restrict__ Yb, int ws, int kw, int wk,
                                              double idv, int lane) {
  if (V >= 2 && wk <= V / 2) {
    trsm_triangle<(V >= 2 ? V / 2 : 1), kScaled>(sm, T, Yb, ws, kw, wk, idv, lane);
    return;
  }
  const int np = (kw + 32 / V - 1) / (32 / V);
  if (np <= 1) trsm_pieces<V, 1, kScaled>(sm, T, Yb, ws, kw, wk, idv, lane);
  else if (V >= 2 && np <= 2) trsm_pieces<V, (V >= 2 ? 2 : 1), kScaled>(sm, T, Yb, ws, kw, wk, idv, lane);
  else if (V >= 4 && np <= 4) trsm_pieces<V, (V >= 4 ? 4 : 1), kScaled>(sm, T, Yb, ws, kw, wk, idv, lane);
  else if (V >= 8 && np <= 8) trsm_pieces<V, (V >= 8 ? 8 : 1), kScaled>(sm, T, Yb, ws, kw, wk, idv, lane);
  else trsm_pieces<V, V, kScaled>(sm, T, Yb, ws, kw, wk, idv, lane);
}

// NJ (row, column) pairs per lane of the update below a block: acc -= L(row, block) X(:, column).
// kFlat: the pairs' columns differ; else they are all col[0].
template <int NJ, bool kFlat, class Sm>
__device__ __forceinline__ void trsm_update(const Sm &sm, const double *__restrict__ Lb, int nr, int kb,
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

// Of listed supernodes l0 .. l0 + 31 those that columns [c_lo, c_hi) reach, into sn; returns how many.
__device__ __forceinline__ int trsm_batch(const PlanPtrs &P, const TrsmTask &t, int l0, int c_lo, int c_hi, TrsmSn *sn,
                                          int lane) {
  bool hit = false;
  SnDev s{};
  if (l0 + lane < t.list_len) {
    s = P.sns[P.trsm_list[t.list_off + l0 + lane]];
    hit = max(s.jlo, c_lo) < min(s.jhi, c_hi);
  }
  const uint32_t m = __ballot_sync(0xffffffffu, hit);
  __syncwarp();
  if (hit) {
    TrsmSn &e = sn[__popc(m & ((1u << lane) - 1))];
    e.y_off = s.y_off; e.rmap_off = s.rmap_off; e.ld_off = s.ld_off; e.lval = P.lcp[s.lcp_off];
    e.ns = s.ns; e.rs = s.rs; e.jlo = s.jlo; e.jhi = s.jhi; e.cut_off = s.cut_off; e.lcp_off = s.lcp_off;
  }
  __syncwarp();
  return __popc(m);
}

// The triangle of a block of kw columns into sm.T by asynchronous copies (Lc[t]: panel row t of column kb).
template <class Sm>
__device__ __forceinline__ void trsm_stage_triangle(Sm &sm, const double *__restrict__ Lc, int nr, int kb, int kw,
                                                    int lane) {
  const double *lp = Lc + kb + lane;
  for (int p = 0; p < kw; ++p) {
    if (lane > p && lane < kw) cp_async8(&sm.T[tri_at(lane, p)], lp, true);
    lp += nr - (kb + p) - 1;
  }
  asm volatile("cp.async.commit_group;\n" ::: "memory");
}

template <int W>
__device__ __forceinline__ void trsm_part(const PlanPtrs &P, const TrsmTask &t, int part,
                                          const double *__restrict__ Lv, const double *__restrict__ invd,
                                          double *__restrict__ Y, TrsmShared<W> &sm, int lane) {
  const int c_lo = t.c_lo + part * W, c_hi = min(c_lo + W, t.c_lo + t.w);
  if (c_lo >= c_hi) return;

  auto batch = [&](int l0) { return trsm_batch(P, t, l0, c_lo, c_hi, sm.sn, lane); };

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
    const int32_t *seed = P.seed_ptr + P.subs[t.sub].col_off;
    const int e1 = seed[c_hi];
    for (int e = seed[c_lo] + lane; e < e1; e += 32) Y[P.seeds[e].y_off] = P.seeds[e].value;
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
          trsm_stage_triangle(sm, Lc, nr, kb, kw, lane);
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
          trsm_triangle<W, false>(sm, sm.T, Yb, ws, kw, wk, idv, lane);
          __syncwarp();
          while (left > 0) {
            switch (min(4, left)) {
              case 1: trsm_update<1, kFlat>(sm, Lc, nr, kb, kw, row, col, acc); break;
              case 2: trsm_update<2, kFlat>(sm, Lc, nr, kb, kw, row, col, acc); break;
              case 3: trsm_update<3, kFlat>(sm, Lc, nr, kb, kw, row, col, acc); break;
              default: trsm_update<4, kFlat>(sm, Lc, nr, kb, kw, row, col, acc); break;
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

}  // namespace sc
