// One query per warp: the 32 lanes of a warp work on one ray or point together.
//
// A launch of few queries ends with the slowest of them, and a query alone in its
// lane is a chain of dependent node loads: 1,000 random points around 50 K
// triangles took 171 us that way, on a GPU that was otherwise idle. Here the
// warp keeps the query's stack in its part of shared memory, takes up to 32 / W
// nodes off its top at a time and tests their W children each, a lane per child
// (or a leaf's triangles, W at a time); what is hit goes back on the stack,
// nearest on top. The chain is as many times shorter. More nodes are visited than
// one after the other, because the best hit so far culls later; the lanes are
// full, which makes up for it until the GPU is (see use_coop in api.cu for where
// the line lies).
//
// Results do not depend on the order of the tests: they are the lexicographic
// minimum of (t, id) or (d2, id), or whether there is a hit.
#pragma once

#include "cpq.cuh"

namespace scion {

// Triangle of leaf entry i.
__device__ __forceinline__ void load_triangle(const TraceArgs &a, uint32_t i, float4 &p0, float4 &p1, float4 &p2,
                                              uint32_t &id) {
  if (a.prim_indirect) {
    id = __ldg(a.prim_ids + i);
    uint32_t v[3];
    for (int k = 0; k < 3; ++k) v[k] = a.tri_idx ? __ldg(a.tri_idx + 3 * (size_t)id + k) : 3 * id + k;
    p0 = ldg4f(a.verts + v[0]);
    p1 = ldg4f(a.verts + v[1]);
    p2 = ldg4f(a.verts + v[2]);
  } else {
    const float4 *q = a.prims + 3 * (size_t)i;
    p0 = ldg4f(q);
    p1 = ldg4f(q + 1);
    p2 = ldg4f(q + 2);
    id = __float_as_uint(p0.w);
  }
}

// Stack entries of a family: the reference of a wide node's child, or an own-box
// node's number. Children per node: kLanes.
template <bool OWN, int W, int PREC, int SOA, int CREF>
struct CoopNode {
  static constexpr uint32_t kLanes = OWN ? 2 : W;
  // Whether entry `ref` is a leaf, with its entries [first, first + count);
  // otherwise `at` is what child() takes.
  static __device__ __forceinline__ bool leaf(const TraceArgs &a, uint32_t ref, uint32_t &first, uint32_t &count,
                                              uint32_t &at) {
    if constexpr (OWN) {
      own_ref<PREC, SOA>(a, ref, count, first);
      at = first;
      return count > 0;
    } else {
      first = ref_leaf_first(ref);
      count = ref_leaf_count(ref);
      at = ref;
      return !ref_is_interior(ref);
    }
  }
  // Child k of the interior entry `ref`: its entry (kEmptyRef: none) and box.
  static __device__ __forceinline__ uint32_t child(const TraceArgs &a, uint32_t ref, uint32_t at, uint32_t k,
                                                   float (&lo)[3], float (&hi)[3]) {
    if constexpr (OWN) {
      const uint32_t l = CREF == REF_DIRECT ? ref + 1 : at, r = CREF == REF_DIRECT ? ref + at : at + 1;
      const uint32_t x = k ? r : l;
      uint32_t c, f;
      own_node<PREC, SOA>(a, x, lo, hi, c, f);
      return x;
    } else {
      using N = WideNode<W, PREC, SOA, CREF>;
      const char *p = reinterpret_cast<const char *>(a.nodes) + (size_t)ref_node(at) * N::kStride;
      uint32_t out;
      if (CREF == REF_DIRECT) {
        out = __ldg(reinterpret_cast<const uint32_t *>(p + N::kRefOff) + k);
      } else {
        const uint32_t *head = reinterpret_cast<const uint32_t *>(p + N::kRefOff);
        const uint8_t *meta = reinterpret_cast<const uint8_t *>(head + 2);
        const uint32_t m = __ldg(meta + k);
        if (m == 0) {
          out = kEmptyRef;
        } else if (m & kMetaInterior) {
          out = ref_interior(__ldg(head) + (m & 0x7Fu));
        } else {
          uint32_t first = __ldg(head + 1);
          for (uint32_t j = 0; j < k; ++j) {
            const uint32_t mj = __ldg(meta + j);
            first += mj & kMetaInterior ? 0u : mj;
          }
          out = ref_leaf(first, m);
        }
      }
      float org[3] = {0.f, 0.f, 0.f}, sc[3] = {1.f, 1.f, 1.f};
      if (N::kGrid) {
        const uint4 h = ldg4(reinterpret_cast<const uint4 *>(p));
        org[0] = __uint_as_float(h.x); org[1] = __uint_as_float(h.y); org[2] = __uint_as_float(h.z);
        sc[0] = __uint_as_float((h.w & 0xFFu) << 23);
        sc[1] = __uint_as_float(((h.w >> 8) & 0xFFu) << 23);
        sc[2] = __uint_as_float(((h.w >> 16) & 0xFFu) << 23);
      }
#pragma unroll
      for (int c = 0; c < 6; ++c) {
        const char *q = p + N::kHdr + (SOA ? c * W + k : k * 6 + c) * N::kElem;
        float v;
        if (PREC == PREC_F32) v = __ldg(reinterpret_cast<const float *>(q));
        else if (PREC == PREC_F16) v = __half2float(__ushort_as_half(__ldg(reinterpret_cast<const unsigned short *>(q))));
        else if (PREC == PREC_U8) v = fmaf((float)__ldg(reinterpret_cast<const unsigned char *>(q)), sc[c % 3], org[c % 3]);
        else v = fmaf((float)__ldg(reinterpret_cast<const unsigned short *>(q)), sc[c % 3], org[c % 3]);
        if (c < 3) lo[c] = v;
        else hi[c - 3] = v;
      }
      return out;
    }
  }
};

// What is asked of the nodes and triangles: a ray's closest hit, whether it has
// any, or the closest point. key: best t or d2 so far.
struct CoopBest {
  float key, u, v;
  uint32_t id;
};

template <bool ANY>
struct CoopRay {
  Ray r;
  __device__ __forceinline__ bool load(const TraceArgs &a, unsigned long long rid, CoopBest &b) {
    const float4 o = ldg4f(a.rays + 2 * rid), d = ldg4f(a.rays + 2 * rid + 1);
    setup_ray(o, d, r);
    b = CoopBest{d.w, 0.f, 0.f, SCION_PRIM_MISS};
    return true;
  }
  static __device__ __forceinline__ float limit(float key) { return far_limit(key); }
  __device__ __forceinline__ bool box(const float (&lo)[3], const float (&hi)[3], float lim, float &key) const {
    return slab(r, lo[0], lo[1], lo[2], hi[0], hi[1], hi[2], lim, key);
  }
  // a triangle that is hit no farther than b
  __device__ __forceinline__ bool triangle(float4 p0, float4 p1, float4 p2, uint32_t id, CoopBest &b) const {
    float t, V, W, det;
    if (!tri_test(r, p0, p1, p2, t, V, W, det)) return false;
    if (ANY) {
      if (!(t <= b.key)) return false;
      b.id = id;
      return true;
    }
    if (!(t < b.key || (t == b.key && id < b.id))) return false;
    b = CoopBest{t, __fdiv_rn(V, det), __fdiv_rn(W, det), id};
    return true;
  }
  static __device__ __forceinline__ void write(const TraceArgs &a, unsigned long long rid, const CoopBest &b) {
    if (ANY) {
      static_cast<uint32_t *>(a.out)[rid] = b.id == SCION_PRIM_MISS ? 0u : (b.id == SCION_PRIM_ERROR ? SCION_PRIM_ERROR : 1u);
    } else {
      const bool none = b.id == SCION_PRIM_MISS || b.id == SCION_PRIM_ERROR;
      static_cast<uint4 *>(a.out)[rid] = make_uint4(none ? 0x7f800000u : __float_as_uint(b.key), __float_as_uint(b.u),
                                                    __float_as_uint(b.v), b.id);
    }
  }
};

struct CoopPoint {
  CpLane L;
  __device__ __forceinline__ bool load(const TraceArgs &a, unsigned long long rid, CoopBest &b) {
    const float4 pt = ldg4f(a.rays + rid);
    L.px = pt.x; L.py = pt.y; L.pz = pt.z;
    b = CoopBest{pt.w, 0.f, 0.f, SCION_PRIM_MISS};
    // a point that is not finite, or a radius that is not >= 0, finds nothing
    return isfinite(pt.x) && isfinite(pt.y) && isfinite(pt.z) && pt.w >= 0.0f;
  }
  static __device__ __forceinline__ float limit(float key) { return cp_limit(key); }
  __device__ __forceinline__ bool box(const float (&lo)[3], const float (&hi)[3], float lim, float &key) const {
    key = box_lower(L, lo[0], lo[1], lo[2], hi[0], hi[1], hi[2]);
    return key <= lim;
  }
  __device__ __forceinline__ bool triangle(float4 p0, float4 p1, float4 p2, uint32_t id, CoopBest &b) const {
    if (!finite_triangle(p0, p1, p2)) return false;
    float u, v;
    const float d2 = cp_triangle(L.px, L.py, L.pz, p0, p1, p2, u, v);
    if (!(d2 < b.key || (d2 == b.key && id < b.id))) return false;
    b = CoopBest{d2, u, v, id};
    return true;
  }
  static __device__ __forceinline__ void write(const TraceArgs &a, unsigned long long rid, const CoopBest &b) {
    CoopRay<false>::write(a, rid, b);
  }
};

// The warp's query `q` from the root; best: its limit, then its result. The same
// in every lane. False: the step limit.
// a.smem_stack entries per lane make a warp's stack of 32 times as many;
// a.stack_need of them are what a tree taken one node at a time can add to it, so
// nodes are taken many at a time only while that much stays free.
template <bool OWN, int W, int PREC, int SOA, int CREF, bool ANY, class Q>
__device__ __forceinline__ bool coop_query(const TraceArgs &a, const Q &q, CoopBest &best, uint2 *stack) {
  using Node = CoopNode<OWN, W, PREC, SOA, CREF>;
  constexpr uint32_t kLanes = Node::kLanes, kGroups = 32 / kLanes;
  const uint32_t lane = threadIdx.x & 31u, g = lane / kLanes, k = lane % kLanes;
  const uint32_t room = 32u * a.smem_stack - a.stack_need - 32u;  // most entries a wide step may start with
  const uint32_t root = OWN ? (a.n_nodes > 0 ? 0u : kEmptyRef) : a.root_ref;
  if (root == kEmptyRef) return true;
  uint32_t sp = 1u, steps = 0;
  if (lane == 0) stack[0] = make_uint2(root, 0xFF800000u);  // key -inf: always entered
  __syncwarp();
  while (sp > 0) {
    const uint32_t n = sp <= room ? min(sp, kGroups) : 1u;
    const bool in = g < n;
    const uint2 e = in ? stack[sp - 1u - g] : make_uint2(kEmptyRef, 0u);
    sp -= n;
    steps += n;
    if (steps > a.max_steps) return false;
    float lim = Q::limit(best.key);
    CoopBest mine = best;
    bool better = false, hit = false;
    uint32_t child = kEmptyRef;
    float key = 0.f;
    if (in && (ANY || __uint_as_float(e.y) <= lim)) {
      uint32_t first, count, at;
      if (Node::leaf(a, e.x, first, count, at)) {
        for (uint32_t i = first + k; i < first + count; i += kLanes) {
          float4 p0, p1, p2;
          uint32_t id;
          load_triangle(a, i, p0, p1, p2, id);
          better |= q.triangle(p0, p1, p2, id, mine);
        }
      } else {
        float lo[3], hi[3];
        child = Node::child(a, e.x, at, k, lo, hi);
        hit = child != kEmptyRef && q.box(lo, hi, lim, key);
      }
    }
    __syncwarp();
    if (__any_sync(0xFFFFFFFFu, better)) {
      if (ANY) {
        best.id = 0u;
        return true;
      }
      // keys are not negative (t >= 0 up to the sign of zero, d2 a sum of
      // squares): their bits order them; -0 counts as 0
      const uint32_t bits = better ? __float_as_uint(mine.key + 0.0f) : 0xFFFFFFFFu;
      const uint32_t low = __reduce_min_sync(0xFFFFFFFFu, bits);
      const uint32_t id = __reduce_min_sync(0xFFFFFFFFu, bits == low ? mine.id : 0xFFFFFFFFu);
      const uint32_t from = __ffs(__ballot_sync(0xFFFFFFFFu, bits == low && mine.id == id && better)) - 1u;
      best.key = __shfl_sync(0xFFFFFFFFu, mine.key, from);
      best.u = __shfl_sync(0xFFFFFFFFu, mine.u, from);
      best.v = __shfl_sync(0xFFFFFFFFu, mine.v, from);
      best.id = id;
      lim = Q::limit(best.key);
      hit = hit && key <= lim;
    }
    const uint32_t hits = __ballot_sync(0xFFFFFFFFu, hit);
    if (hits) {
      uint32_t rank = 0;  // places above the stack: farther entries below
      if (ANY) {
        rank = __popc(hits & ((1u << lane) - 1u));
      } else {
        for (uint32_t m = hits; m; m &= m - 1u) {
          const uint32_t j = __ffs(m) - 1u;
          const float other = __shfl_sync(0xFFFFFFFFu, key, j);
          rank += other > key || (other == key && j < lane) ? 1u : 0u;
        }
      }
      if (hit) stack[sp + rank] = make_uint2(child, __float_as_uint(key));
      sp += __popc(hits);
    }
    __syncwarp();
  }
  return true;
}

template <bool OWN, int W, int PREC, int SOA, int CREF, bool ANY, class Q>
__device__ __forceinline__ void coop_body(const TraceArgs &a) {
  extern __shared__ uint2 smem_stack[];
  uint2 *const stack = smem_stack + (threadIdx.x & ~31u) * a.smem_stack;
  const uint32_t lane = threadIdx.x & 31u;
  for (unsigned long long block = first_block(); block < a.n_work; block = take_block(a)) {  // chunk = 1
    const unsigned long long rid = slot_ray(a, block);
    if (rid >= a.n) continue;  // the same for the whole warp
    Q q;
    CoopBest best;
    if (q.load(a, rid, best) && !coop_query<OWN, W, PREC, SOA, CREF, ANY>(a, q, best, stack)) {
      if (lane == 0) atomicCAS(a.status, 0u, kErrIter);
      best = CoopBest{0.f, 0.f, 0.f, SCION_PRIM_ERROR};
    }
    if (lane == 0) Q::write(a, rid, best);
    __syncwarp();
  }
  release_blocks(a);
}

}  // namespace scion
