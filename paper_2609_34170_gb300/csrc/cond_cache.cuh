// The check of the conditioning cache (device code without CUDA headers' device
// functions beyond atomicOr and __syncthreads, so that it compiles for the host
// too).
#pragma once

#include "kernels.h"

namespace ravel {

// Which rows of this step's conditioning are cached already (see CondCache).
// The slot times hit when every one equals the cached key; a robot's offset
// hits when its value is one of the cached offsets.  Misses get a cache slot (a
// slot already referenced in this step is never taken; with no slot left the
// robot keeps this step's fresh row), and their keys are written now: the rows
// themselves arrive through cond_commit before any reader of this step, and a
// later step reads them only after that.  One block; bound by load latency, so
// every key is read once, in parallel, and the loop over the robots runs only
// where one misses (that loop and one key after the other took 64 robots 3 us
// more, hit or miss).
// t_key holds the slot times of one schedule (slots floats) and is touched only
// where the cache is on; with a schedule per robot H is B slots and the cache off.
__device__ inline void cond_check(const CondArgs& a) {
  __shared__ int s_tmiss, s_bmiss, s_used[kCondCache];
  __shared__ float s_key[kCondCache];
  __shared__ unsigned s_ref;   // cache slots referenced by this step
  CondCache* cc = a.cc;
  if (threadIdx.x < kCondCache) {
    s_used[threadIdx.x] = cc->used[threadIdx.x];
    s_key[threadIdx.x] = cc->delta[threadIdx.x];
  }
  if (threadIdx.x == 0) {
    s_tmiss = a.enabled && !a.fresh ? !cc->t_valid : 1;
    s_bmiss = 0;
    s_ref = 0u;
  }
  __syncthreads();
  if (a.enabled && !a.fresh)
    for (int j = threadIdx.x; j < a.H; j += blockDim.x)
      if (a.slot_times[j] != a.t_key[j]) s_tmiss = 1;   // benign race: every writer stores 1
  // offsets: look up in parallel; -1 = miss
  for (int b = threadIdx.x; b < a.B; b += blockDim.x) {
    int row = a.enabled ? -1 : a.H + b;
    if (a.enabled) {
      const float d = a.delta[b];
      for (int c = 0; c < kCondCache; ++c)
        if (s_used[c] && s_key[c] == d) {
          row = a.H + a.Bmax + c;
          atomicOr(&s_ref, 1u << c);
          break;
        }
      if (row < 0) s_bmiss = 1;
    }
    a.drow[b] = row;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    int nc = 0;
    unsigned ref = s_ref;
    for (int b = 0; s_bmiss && b < a.B; ++b) {
      if (a.drow[b] >= 0) continue;
      const float d = a.delta[b];
      int row = a.H + b;   // this step's fresh row unless a cache slot is found
      int c = -1;
      for (int k = 0; k < kCondCache; ++k)   // assigned to an earlier robot of this step?
        if ((ref >> k & 1u) && cc->used[k] && cc->delta[k] == d) c = k;
      if (c < 0) {
        for (int k = 0; k < kCondCache && c < 0; ++k) {
          const int v = (cc->next + k) % kCondCache;
          if (!(ref >> v & 1u)) c = v;
        }
        if (c >= 0) {
          cc->next = (c + 1) % kCondCache;
          cc->delta[c] = d;
          cc->used[c] = 1;
          a.commit[2 * nc] = a.H + b;
          a.commit[2 * nc + 1] = a.H + a.Bmax + c;
          ++nc;
        }
      }
      if (c >= 0) {
        ref |= 1u << c;
        row = a.H + a.Bmax + c;
      }
      a.drow[b] = row;
    }
    cc->n_commit = nc;
    cc->skip = s_tmiss || s_bmiss ? 0 : 1;
    if (a.enabled) cc->t_valid = 1;
  }
  // the slot times become the key (a miss recomputes rows [0, H) this step)
  if (a.enabled)
    for (int j = threadIdx.x; j < a.H; j += blockDim.x) a.t_key[j] = a.slot_times[j];
}

}  // namespace ravel
