// Body of the multi-scene kernel for scenes of one node family (see batched.cu).
#pragma once

#include "batched.h"

namespace scion {

template <bool OWN, int W, int PREC, int SOA>
__device__ __forceinline__ void batched_body(const BatchArgs &ba) {
  extern __shared__ uint2 smem_stack[];
  // per warp (256 threads at most): the scene it is at and the slots it has.
  // Registers are what this kernel is short of.
  struct At {
    TraceArgs a;
    unsigned long long begin, end;
  };
  __shared__ At scene_at[8];
  StackFor<OWN, PREC, W, false, 0> st;
  StackTail<decltype(st)::kTF, decltype(st)::kKeyed> tail;
  st.attach(tail);
  st.columns(smem_stack, ba.smem_stack);
  st.reset();
  TraceQuery<OWN, W, PREC, SOA, REF_DIRECT, false, false, decltype(st)> q(st);
  const uint32_t lane = threadIdx.x & 31u, below = (1u << lane) - 1u;
  At &at = scene_at[threadIdx.x >> 5];
  const TraceArgs &a = at.a;
  // the unit numbers of a batch fit 32 bits (2^32 units of 32 rays are more
  // than the device holds)
  auto units = [&]() { return (uint32_t)(ba.slots / ba.chunk); };
  auto counted = [&]() { return units() > grid_warps(); };  // otherwise every unit has a warp of its own
  auto take = [&]() {
    if (!counted()) return units();
    uint32_t u = 0;
    if (lane == 0) u = (uint32_t)(atomicAdd(ba.work, 1ull) + grid_warps());
    return __shfl_sync(0xFFFFFFFFu, u, 0);
  };
  uint32_t unit = (uint32_t)first_block();
  while (unit < units()) {
    // the last scene that begins at or before the unit
    const unsigned long long slot0 = (unsigned long long)unit * ba.chunk;
    uint32_t lo = 0, hi = ba.n_scenes;
    while (hi - lo > 1) {
      const uint32_t mid = (lo + hi) >> 1;
      if (__ldg(&ba.scenes[mid].begin) <= slot0) lo = mid;
      else hi = mid;
    }
    __syncwarp();  // every lane is done with the last scene's arguments
    const uint32_t *src = reinterpret_cast<const uint32_t *>(&ba.scenes[lo].a);
    for (uint32_t i = lane; i < sizeof(TraceArgs) / 4; i += 32) reinterpret_cast<uint32_t *>(&at.a)[i] = __ldg(src + i);
    if (lane == 0) {
      at.begin = __ldg(&ba.scenes[lo].begin);
      at.end = at.begin + ((__ldg(&ba.scenes[lo].a.n) + 31ull) & ~31ull);
    }
    __syncwarp();
    if (ba.chunk < 32u || a.refill_min >= 32u) {
      do {
        const unsigned long long rid = (unsigned long long)unit * ba.chunk - at.begin + lane;
        if (lane < ba.chunk && rid < a.n) {
          q.start(a, rid);
          while (q.busy()) q.step(a);
          q.finish(a);
        }
        unit = take();
      } while ((unsigned long long)unit * ba.chunk < at.end);
      continue;
    }
    uint32_t taken = 0;   // slots of the unit handed out
    bool mine = true;     // the unit belongs to this scene
    bool holds = false;   // this lane has a ray whose result is not written
    q.idle();
    while (true) {
      const uint32_t idle = __ballot_sync(0xFFFFFFFFu, !q.busy());
      if ((uint32_t)__popc(idle) >= a.refill_min) {
        if (holds && !q.busy()) {
          q.finish(a);
          holds = false;
        }
        if (taken >= 32u && mine) {
          unit = take();
          taken = 0;
          mine = unit * 32ull < at.end;
        }
        if (mine) {
          if (!q.busy()) {
            const uint32_t i = taken + __popc(idle & below);
            const unsigned long long rid = unit * 32ull - at.begin + i;
            if (i < 32u && rid < a.n) {
              q.start(a, rid);
              holds = true;
            }
          }
          taken += __popc(idle);
        } else if (idle == 0xFFFFFFFFu) {
          break;
        }
      }
#pragma unroll 1
      for (int j = 0; j < kFreeSteps && q.busy(); ++j) q.step(a);
    }
  }
  if (!counted()) return;
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    const uint32_t prev = atomicAdd(ba.exit_count, 1u);
    if (prev == gridDim.x - 1) {
      *ba.work = 0ull;
      *ba.exit_count = 0u;
      __threadfence();
    }
  }
}

}  // namespace scion
