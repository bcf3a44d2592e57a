// sm_103a kernels of the Schur-complement assembly and application (FP64).
//
//   prep_kernel   -- reciprocal of L's diagonal for every column of an active
//                    supernode; a non-positive / non-finite pivot sets the
//                    NOT_SPD bit of the workspace status word (paper Sec. 3.1:
//                    the factor is copied in; here its CSC columns are read
//                    in place, because a fundamental supernode's CSC column is
//                    already a dense trapezoidal panel column); F's padding,
//                    and for split precision Y's column bounds and a look at
//                    the triangles' range.
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
#include "sc_trsm.cuh"

namespace sc {

// One launch for what the stages need beforehand (two launches cost a small batch
// 3 us of its 60).  CTAs below nprep: reciprocal diagonal.  The next, one per
// subdomain: zero the entries of F beyond m (rows >= m of the last tile row and
// columns >= m of the last diagonal tile).  The others, for split precision: zero the column bounds of Y and
// look at the triangles, a warp to a (supernode, block).  Where an entry is so far from its column's diagonal (rows of L
// that differ by hundreds of orders of magnitude) that FP64 may not hold their ratio in full, the
// split TRSM must not divide its triangles by the diagonal.
template <bool kSplit>
__global__ void __launch_bounds__(256) prep_kernel(const int64_t *__restrict__ lcp, const int32_t *__restrict__ active,
                                                   int64_t nact, int nprep, const double *__restrict__ Lv,
                                                   double *__restrict__ invd, uint32_t *__restrict__ status,
                                                   const SubDev *__restrict__ subs, int nsub, double *__restrict__ F,
                                                   const PlanPtrs P, int64_t nsblk, int *__restrict__ colexp,
                                                   int64_t ncols) {
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
  if (kSplit && (int)blockIdx.x >= nprep + nsub) {
    const int64_t cta = blockIdx.x - nprep - nsub, nt = (int64_t)(gridDim.x - nprep - nsub) * blockDim.x;
    for (int64_t k = cta * blockDim.x + threadIdx.x; k < ncols; k += nt) colexp[k] = 0;
    const int64_t item = cta * (blockDim.x / 32) + threadIdx.x / 32;
    if (item >= nsblk) return;
    const SnDev s = P.sns[P.sblk[2 * item]];
    const int kb = 32 * P.sblk[2 * item + 1], kw = min(32, s.ns - kb), nr = s.ns + s.rs - kb, r = threadIdx.x & 31;
    if (kw <= kDirect) return;
    // high words; entry (t, q) of the triangle at q nr - q (q + 1) / 2 + t
    const uint32_t *Lh = reinterpret_cast<const uint32_t *>(Lv + lcp[s.lcp_off + kb]) + 1;
    bool out = false;
#pragma unroll 8
    for (int q = 0; q < kw; ++q) {
      const int o = q * nr - q * (q + 1) / 2;
      const uint32_t l = r > q && r < kw ? Lh[2 * (o + r)] : 0u, d = r > q && r < kw ? Lh[2 * (o + q)] : 0u;
      const int e = (int)(l >> 20 & 0x7FFu), f = e - (int)(d >> 20 & 0x7FFu);
      out |= (l << 1 != 0u) & ((e == 0) | (f < -1020) | (f > 1020));
    }
    if (out) status[kUnscaledWord] = 1u;
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
  int64_t ncols = 0, ncheck = 0;
  if (c.n_slices > 0) {
    for (int32_t m : c.m) ncols += m;
    ncheck = std::max<int64_t>((c.n_sblk + 7) / 8, ncols > 0);
  }
  if (nprep + c.nsub > 0) {
    auto kernel = c.n_slices > 0 ? prep_kernel<true> : prep_kernel<false>;
    kernel<<<(unsigned)(nprep + c.nsub + ncheck), 256, 0, S(stream)>>>(
        p.lcp, p.active_cols, c.n_active_cols, nprep, Lv, invd, status, p.subs, c.nsub, F, p, c.n_sblk,
        reinterpret_cast<int *>(static_cast<uint8_t *>(ws) + c.ws.colexp_off), ncols);
  }
  return (int)cudaGetLastError();
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
      switch (G.trsm_cols[0]) {
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
  if (!e) e = launch_trsm_split(c, S, G.trsm_cols[v], G.trsm[v][0], G.trsm[v][1], Lv, invd, ws, Y, stream);
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
