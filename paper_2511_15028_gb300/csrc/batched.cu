// Many scenes in one persistent launch (closest hit).
//
// Every scene keeps its own BVH and layout. Its rays occupy a range of a global
// index space padded to multiples of 32, so each unit a warp takes from the
// global counter belongs to exactly one scene; the warp stays with the scene
// while the next units it takes belong to it. The scene's fetch mode holds:
// warp batches (each lane traces its ray of the unit to completion, then the
// warp takes the next unit) or warp refill (idle lanes take the next rays as
// soon as at least rays_per_fetch of them are idle, from a new unit when the
// current one is used up; a unit of another scene ends the refill, the warp
// finishes its rays and moves on).
//
// Where all scenes have one node family, as an autotuned batch usually does, a
// kernel of that family runs (batched_body in batched.cuh, instantiated beside
// the family's other kernels): its loops are the plain launch's, with the
// scene's arguments in shared memory. A batch of several families with enough
// rays is launched a family at a time (split_batch in api.cu); a smaller one runs in
// the kernel below, which dispatches with a warp-uniform switch over functions of
// their own; those spill 200 to 300 bytes under the 64-register cap and read the
// scene's arguments from global memory, which is why it is not used for both.
// Measured, 48 scenes of one family (1.6 M rays): bvh4 u8 batches 839 -> 775 us,
// refill 1,319 -> 847; bvh4 f32 refill 1,342 -> 854; bvh8 u8 1,131 -> 954; bvh2 q16
// refill 2,511 -> 1,198; 5 small scenes 121 -> 68 (48 scenes, bvh4 u8, with the
// steps of node_then_leaf: 707). One large scene runs within 4 %
// of its plain launch (refill: twice as long before).
// The launch allocates nothing and never synchronises the host, so it can be
// captured in a CUDA graph and replayed; its counters reset themselves.
#include <cuda_runtime.h>

#include "batched.h"
#include "kernels.h"

namespace scion {

namespace {

constexpr int kMaxSharedScenes = 1024;  // scene starts cached in shared memory

// One visit per step: the steps of node_then_leaf spill 30 to 60 % more here
// (64 scenes of three families, 7.2 M rays: 4.39 -> 3.79 to 4.16 ms).
template <bool OWN, int W, int PREC, int SOA>
__device__ __forceinline__ void step_family(const TraceArgs &a, Lane &L, Stack &st, Counts &cnt) {
  if constexpr (OWN) {
    if (L.count > 0) leaf_bin<PREC, SOA, false, false>(a, L, st, cnt);
    else node_bin<PREC, SOA, REF_DIRECT, false, false>(a, L, st, cnt);
  } else {
    if (ref_is_interior(L.cur)) node_wide<W, PREC, SOA, REF_DIRECT, false, false>(a, L, st, cnt);
    else leaf_wide<false, false>(a, L, st, cnt);
  }
  if (L.steps > a.max_steps) {
    L.err = kErrIter;
    L.cur = kEmptyRef;
  }
}

// The next 32-ray unit of the global index space (warp-uniform).
__device__ __forceinline__ unsigned long long take_unit(unsigned long long *work) {
  unsigned long long b = 0;
  if ((threadIdx.x & 31u) == 0) b = atomicAdd(work, (unsigned long long)kBatchUnit);
  return __shfl_sync(0xFFFFFFFFu, b, 0);
}

template <bool OWN, int PREC, int SOA>
__device__ __forceinline__ void start_lane(const TraceArgs &a, Lane &L, Stack &st, unsigned long long rid) {
  L.rid = rid;
  const float4 o = ldg4f(a.rays + 2 * rid), d = ldg4f(a.rays + 2 * rid + 1);
  setup_ray(o, d, L.r);
  L.b = Best{d.w, 0.f, 0.f, SCION_PRIM_MISS};
  L.steps = 0;
  L.err = 0;
  L.found = false;
  st.reset();
  start_ray<OWN, PREC, SOA>(a, L);
}

__device__ __forceinline__ void finish_lane(const TraceArgs &a, Lane &L) {
  if (L.err) {
    atomicCAS(a.status, 0u, L.err);
    L.b = Best{__int_as_float(0x7f800000), 0.f, 0.f, SCION_PRIM_ERROR};
  }
  if (L.b.id == SCION_PRIM_MISS) L.b.t = __int_as_float(0x7f800000);
  static_cast<uint4 *>(a.out)[L.rid] =
      make_uint4(__float_as_uint(L.b.t), __float_as_uint(L.b.u), __float_as_uint(L.b.v), L.b.id);
}

// Trace the scene's unit at `base` and every following unit the warp takes
// while they belong to the scene; returns the first unit taken that does not
// (another scene's, or >= total). Not inlined: each family's loops get their
// own register allocation (inlined into one switch they spill heavily); the
// call costs once per scene change of a warp.
// The stack is made here, not passed in: an object whose address crosses a
// call lives in local memory, and so would the stack pointer on every step.
template <bool OWN, int W, int PREC, int SOA>
__device__ __noinline__ unsigned long long run_scene(const BatchScene &S, unsigned long long base,
                                                     unsigned long long *work, uint2 *smem_base,
                                                     uint32_t smem_stack) {
  Stack st;
  StackTail<false> tail;
  st.attach(tail);
  st.columns(smem_base, smem_stack);
  st.reset();
  const TraceArgs &a = S.a;
  const unsigned long long s_lo = S.begin, s_hi = S.begin + ((a.n + 31ull) & ~31ull);
  const uint32_t lane = threadIdx.x & 31u;
  Counts cnt;
  Lane L;
  if (a.refill_min == 32) {
    // warp batches: every lane traces its ray of the unit to completion
    while (base >= s_lo && base < s_hi) {
      const unsigned long long rid = base - s_lo + lane;
      if (rid < a.n) {
        start_lane<OWN, PREC, SOA>(a, L, st, rid);
        while (L.cur != kEmptyRef) step_family<OWN, W, PREC, SOA>(a, L, st, cnt);
        finish_lane(a, L);
      }
      base = take_unit(work);
    }
    return base;
  }
  // warp refill from the rays [next, hi) of the current unit
  const uint32_t k = a.refill_min;
  const uint32_t below = (1u << lane) - 1u;  // lanes ranked before this one
  unsigned long long next = base - s_lo;
  unsigned long long hi = next + kBatchUnit < a.n ? next + kBatchUnit : a.n;
  unsigned long long pending = 0;
  bool mine = true;  // the last unit taken belongs to this scene
  bool has_ray = false;
  L.cur = kEmptyRef;
  while (true) {
    const uint32_t idle = __ballot_sync(0xFFFFFFFFu, !has_ray);
    const uint32_t n_idle = __popc(idle);
    if (n_idle >= k) {
      if (next >= hi && mine) {
        const unsigned long long b = take_unit(work);
        if (b >= s_lo && b < s_hi) {
          next = b - s_lo;
          hi = next + kBatchUnit < a.n ? next + kBatchUnit : a.n;
        } else {
          mine = false;
          pending = b;
        }
      }
      if (next < hi) {
        if (!has_ray) {
          const unsigned long long rid = next + __popc(idle & below);
          if (rid < hi) {
            start_lane<OWN, PREC, SOA>(a, L, st, rid);
            has_ray = true;
          }
        }
        next = next + n_idle < hi ? next + n_idle : hi;
      }
    }
    // a unit of this scene always holds a ray, so with every lane idle the
    // warp either took rays above or has moved past the scene
    if (__ballot_sync(0xFFFFFFFFu, has_ray) == 0u) break;
    if (has_ray && L.cur != kEmptyRef) step_family<OWN, W, PREC, SOA>(a, L, st, cnt);
    if (has_ray && L.cur == kEmptyRef) {
      finish_lane(a, L);
      has_ray = false;
    }
  }
  return pending;
}

__global__ void __launch_bounds__(kMaxThreadsPerBlock, kMinBlocksPerSm)
    batched_kernel(BatchArgs ba) {
  const BatchScene *__restrict__ scenes = ba.scenes;
  const uint32_t n_scenes = ba.n_scenes, smem_stack = ba.smem_stack;
  const unsigned long long total = ba.slots;
  unsigned long long *const work = ba.work;
  uint32_t *const exit_count = ba.exit_count;
  extern __shared__ uint2 smem[];
  // scene starts (padded global offsets) for the unit -> scene search
  __shared__ unsigned long long starts[kMaxSharedScenes];
  const uint32_t cached = n_scenes < (uint32_t)kMaxSharedScenes ? n_scenes : (uint32_t)kMaxSharedScenes;
  for (uint32_t i = threadIdx.x; i < cached; i += blockDim.x) starts[i] = scenes[i].begin;
  __syncthreads();
  unsigned long long base = take_unit(work);
  while (base < total) {
    // last scene whose start <= base (binary search, warp-uniform)
    uint32_t lo = 0, hi = n_scenes;
    while (hi - lo > 1) {
      const uint32_t mid = (lo + hi) >> 1;
      const unsigned long long sm = mid < cached ? starts[mid] : scenes[mid].begin;
      if (sm <= base) lo = mid;
      else hi = mid;
    }
    const BatchScene &S = scenes[lo];
    switch (S.family) {
      case kFamilyBin: base = run_scene<true, 2, PREC_F32, LAYOUT_AOS>(S, base, work, smem, smem_stack); break;
      case kFamilyBinQ16: base = run_scene<true, 2, PREC_Q16, LAYOUT_AOS>(S, base, work, smem, smem_stack); break;
      case kFamilyW4F32: base = run_scene<false, 4, PREC_F32, LAYOUT_SOA>(S, base, work, smem, smem_stack); break;
      case kFamilyW4F16: base = run_scene<false, 4, PREC_F16, LAYOUT_SOA>(S, base, work, smem, smem_stack); break;
      case kFamilyW4U8: base = run_scene<false, 4, PREC_U8, LAYOUT_SOA>(S, base, work, smem, smem_stack); break;
      case kFamilyW8F16: base = run_scene<false, 8, PREC_F16, LAYOUT_SOA>(S, base, work, smem, smem_stack); break;
      case kFamilyW8U8: base = run_scene<false, 8, PREC_U8, LAYOUT_AOS>(S, base, work, smem, smem_stack); break;
      case kFamilyW8U8S: base = run_scene<false, 8, PREC_U8, LAYOUT_SOA>(S, base, work, smem, smem_stack); break;
      default: base = take_unit(work); break;  // batch creation admits only the families above
    }
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    const uint32_t prev = atomicAdd(exit_count, 1u);
    if (prev == gridDim.x - 1) {
      *work = 0ull;
      *exit_count = 0u;
      __threadfence();
    }
  }
}

}  // namespace

int batched_family(uint32_t own_box, const scion_layout_desc &d) {
  if (d.child_ref != REF_DIRECT) return -1;
  if (own_box) {
    if (d.box_layout != LAYOUT_AOS) return -1;
    if (d.box_prec == PREC_F32) return (int)kFamilyBin;
    if (d.box_prec == PREC_Q16) return (int)kFamilyBinQ16;
    return -1;
  }
  if (d.width == 4 && d.box_layout == LAYOUT_SOA) {
    if (d.box_prec == PREC_F32) return (int)kFamilyW4F32;
    if (d.box_prec == PREC_F16) return (int)kFamilyW4F16;
    if (d.box_prec == PREC_U8) return (int)kFamilyW4U8;
    return -1;
  }
  if (d.width == 8 && d.box_prec == PREC_F16 && d.box_layout == LAYOUT_SOA) return (int)kFamilyW8F16;
  if (d.width == 8 && d.box_prec == PREC_U8) return d.box_layout == LAYOUT_AOS ? (int)kFamilyW8U8 : (int)kFamilyW8U8S;
  return -1;
}

BatchKernel batched_kernel_for(int family) {
  switch (family) {
    case kFamilyBin: return batched_own_p0(LAYOUT_AOS);
    case kFamilyBinQ16: return batched_own_p3(LAYOUT_AOS);
    case kFamilyW4F32: return batched_w4_p0(LAYOUT_SOA);
    case kFamilyW4F16: return batched_w4_p1(LAYOUT_SOA);
    case kFamilyW4U8: return batched_w4_p2(LAYOUT_SOA);
    case kFamilyW8F16: return batched_w8_p1(LAYOUT_SOA);
    case kFamilyW8U8: return batched_w8_p2(LAYOUT_AOS);
    case kFamilyW8U8S: return batched_w8_p2(LAYOUT_SOA);
    default: return batched_kernel;
  }
}

}  // namespace scion
