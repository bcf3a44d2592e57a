// Walking the stored 32x32 tiles of every F_i in storage order (subdomain, row block I, J = 0 .. I).
#pragma once

#include <cstdint>

#include "sc_internal.h"

namespace sc {

// the first tile of apply task k (storage order: subdomain, row block I, J = 0..I)
__device__ __forceinline__ int64_t task_tile0(const PlanPtrs &P, int64_t k) {
  const ApplyTask a = P.apply_tasks[k];
  return P.subs[a.sub].F_off / 1024 + (int64_t)a.I * (a.I + 1) / 2;
}

struct TileCursor {
  int64_t task;
  int sub, I, J, m;
  __device__ __forceinline__ void load(const PlanPtrs &P) {
    const ApplyTask a = P.apply_tasks[task];
    sub = a.sub;
    I = a.I;
    m = P.subs[a.sub].m;
  }
  __device__ __forceinline__ void next(const PlanPtrs &P) {
    if (++J > I) {
      ++task;
      J = 0;
      load(P);
    }
  }
};

// The cursor at tile t0 < the number of tiles (a whole warp calls it): 32 tasks are probed at a time, since
// every probe is two dependent loads.
__device__ __forceinline__ TileCursor tile_at(const PlanPtrs &P, int64_t n_tasks, int64_t t0) {
  const int lane = threadIdx.x & 31;
  int64_t lo = 0, hi = n_tasks - 1;               // the task holding tile t0 is one of lo .. hi
  while (lo < hi) {
    const int64_t step = (hi - lo + 31) / 32, k = lo + (lane + 1) * step;
    lo += step * __popc(__ballot_sync(0xffffffffu, k <= hi && task_tile0(P, k) <= t0));
    hi = lo + step - 1 < hi ? lo + step - 1 : hi;
  }
  TileCursor cur{lo, 0, 0, 0, 0};
  cur.load(P);
  cur.J = (int)(t0 - task_tile0(P, lo));
  return cur;
}

}  // namespace sc
