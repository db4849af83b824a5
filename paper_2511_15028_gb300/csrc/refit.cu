// Refit: new vertex positions, same tree. See refit.h.
//
// Works on the packed tree itself, so every layout refits without any host
// state: (1) the vertex table and the direct triangle copies are rewritten;
// (2) on the first refit of a BVH each node's parent and its number of interior
// children are read off the packed references (the tree never changes, so
// they stay); (3) each node's box over its own leaves, then exact boxes
// bottom-up: a thread starts at every node without interior children and
// climbs while it is the last child to arrive at a node (an atomic counter,
// which that thread sets back for the next refit; nothing waits); (4) the world
// grid of q16/eq10 is recomputed from the new root box; (5) every node
// re-encodes its box fields, byte for byte as the packers write them.
//
// Bound by memory latency and by the encoders' arithmetic: for 1.4 M triangles
// the buffers that must be read and written (vertices, triangle copies, node
// boxes) are 0.15 GB, 22 us at the measured copy bandwidth. The kernels are
// compiled per node width, so children stay in registers (one kernel for
// every layout kept them in local memory), leaf boxes are computed for all
// nodes at once and not on the way up, where few lanes of a warp are left,
// and the encoders run in FP32 (codec_fast.h) and write through shared
// memory. Measured for 1.4 M triangles, refit and a 720p frame traced after it:
// bvh8 u8 1.32 -> 0.51 ms (0.28 of it the trace; encoder 0.81 -> 0.11), bvh4 f32
// 0.93 -> 0.41, bvh2 q16 1.24 -> 0.65; 20 K triangles 0.26 -> 0.09.
#include "refit.h"

#include "codec_fast.h"

namespace scion {

namespace {

constexpr uint32_t kNoParent = 0xFFFFFFFFu;
constexpr int kEncodeThreads = 128;

struct Tree {
  uint8_t *nodes;
  const uint8_t *nodes2;
  float4 *prims;            // direct triangle copies (or null)
  const uint32_t *prim_ids; // indirect entries (or null)
  float4 *verts;            // float4 vertex table
  const uint32_t *tri_idx;  // u32[3] per triangle, or null for a soup
  uint32_t n_nodes, stride, prec, soa, cref;
};

__device__ __forceinline__ Box3 empty_box() {
  Box3 b;
  for (int a = 0; a < 3; ++a) {
    b.lo[a] = INFINITY;
    b.hi[a] = -INFINITY;
  }
  return b;
}

__device__ __forceinline__ void grow(Box3 &b, const Box3 &c) {
  for (int a = 0; a < 3; ++a) {
    b.lo[a] = fminf(b.lo[a], c.lo[a]);
    b.hi[a] = fmaxf(b.hi[a], c.hi[a]);
  }
}

__device__ __forceinline__ void triangle_verts(const Tree &t, uint32_t id, uint32_t (&i)[3]) {
  if (t.tri_idx) {
    for (int k = 0; k < 3; ++k) i[k] = __ldg(t.tri_idx + 3 * (size_t)id + k);
  } else {
    for (int k = 0; k < 3; ++k) i[k] = 3 * id + k;
  }
}

// exact box of the leaf entries [first, first + count); triangles with a
// non-finite vertex are left out (they are never hit)
__device__ __forceinline__ Box3 leaf_box(const Tree &t, uint32_t first, uint32_t count) {
  Box3 b = empty_box();
  for (uint32_t e = first; e < first + count; ++e) {
    float4 p[3];
    if (t.prims) {
      for (int k = 0; k < 3; ++k) p[k] = t.prims[3 * (size_t)e + k];
    } else {
      uint32_t i[3];
      triangle_verts(t, __ldg(t.prim_ids + e), i);
      for (int k = 0; k < 3; ++k) p[k] = t.verts[i[k]];
    }
    bool finite = true;
    for (int k = 0; k < 3; ++k) finite &= isfinite(p[k].x) && isfinite(p[k].y) && isfinite(p[k].z);
    if (!finite) continue;
    for (int k = 0; k < 3; ++k) {
      b.lo[0] = fminf(b.lo[0], p[k].x); b.hi[0] = fmaxf(b.hi[0], p[k].x);
      b.lo[1] = fminf(b.lo[1], p[k].y); b.hi[1] = fmaxf(b.hi[1], p[k].y);
      b.lo[2] = fminf(b.lo[2], p[k].z); b.hi[2] = fmaxf(b.hi[2], p[k].z);
    }
  }
  return b;
}

// boxes are 24 bytes, 8-byte aligned; read past L1 (other SMs write them)
__device__ __forceinline__ Box3 load_box(const Box3 *boxes, uint32_t i) {
  const float2 *f = reinterpret_cast<const float2 *>(boxes + i);
  const float2 a = __ldcg(f), b = __ldcg(f + 1), c = __ldcg(f + 2);
  Box3 r;
  r.lo[0] = a.x; r.lo[1] = a.y; r.lo[2] = b.x;
  r.hi[0] = b.y; r.hi[1] = c.x; r.hi[2] = c.y;
  return r;
}
__device__ __forceinline__ void store_box(Box3 *boxes, uint32_t i, const Box3 &b) {
  float2 *f = reinterpret_cast<float2 *>(boxes + i);
  f[0] = make_float2(b.lo[0], b.lo[1]);
  f[1] = make_float2(b.lo[2], b.hi[0]);
  f[2] = make_float2(b.hi[1], b.hi[2]);
}

// ------------------------------------------------------------ own-box nodes
// reference and primitive count (0: interior) of own-box node x
__device__ __forceinline__ void own_slot(const Tree &t, uint32_t x, uint32_t &field, uint32_t &count) {
  const uint8_t *p = t.nodes + (size_t)x * t.stride;
  if (t.prec == PREC_SLAB || t.prec == PREC_F32) {
    const uint8_t *q = t.prec == PREC_SLAB ? p + 8 : (t.soa ? t.nodes2 + (size_t)x * kBinRefBytes : p + 24);
    field = *reinterpret_cast<const uint32_t *>(q);
    count = bin_meta_count(*reinterpret_cast<const uint32_t *>(q + 4));
  } else {
    const uint32_t w = *reinterpret_cast<const uint32_t *>(
        t.prec == PREC_Q16 ? (t.soa ? t.nodes2 + (size_t)x * 4 : p + 12) : p + 8);
    count = qbin_count(w);
    field = count > 0 ? qbin_first(w) : qbin_field(w);
  }
}

// A family of nodes: its interior children (in kids, n of them) and the box
// over its leaves. W = 0: own-box binary nodes, whose leaves are nodes.
template <int W>
struct Family {
  static constexpr int kKids = W == 0 ? 2 : W;
  // references of a wide node's children as direct references
  static __device__ __forceinline__ void refs(const Tree &t, uint32_t x, uint32_t (&r)[kKids]) {
    const uint32_t off = wide_ref_offset(W, t.prec);
    const uint8_t *p = t.nodes + (size_t)x * t.stride + off;
    if (t.cref == REF_DIRECT) {
      for (int k = 0; k < W; ++k) r[k] = *reinterpret_cast<const uint32_t *>(p + 4 * k);
      return;
    }
    const uint32_t base_node = *reinterpret_cast<const uint32_t *>(p);
    uint32_t at = *reinterpret_cast<const uint32_t *>(p + 4);
    for (int k = 0; k < W; ++k) {
      const uint32_t m = p[8 + k];
      if (m & kMetaInterior) {
        r[k] = ref_interior(base_node + (m & 0x7Fu));
      } else if (m) {
        r[k] = ref_leaf(at, m);
        at += m;
      } else {
        r[k] = kEmptyRef;
      }
    }
  }
  static __device__ __forceinline__ uint32_t ref(const Tree &t, uint32_t x, uint32_t k) {
    const uint8_t *p = t.nodes + (size_t)x * t.stride + wide_ref_offset(W, t.prec);
    if (t.cref == REF_DIRECT) return *reinterpret_cast<const uint32_t *>(p + 4 * k);
    const uint32_t m = p[8 + k];
    if (m == 0) return kEmptyRef;
    if (m & kMetaInterior) return ref_interior(*reinterpret_cast<const uint32_t *>(p) + (m & 0x7Fu));
    uint32_t at = *reinterpret_cast<const uint32_t *>(p + 4);
    for (uint32_t i = 0; i < k; ++i) at += p[8 + i] & kMetaInterior ? 0u : p[8 + i];
    return ref_leaf(at, m);
  }
  static __device__ __forceinline__ uint32_t kids(const Tree &t, uint32_t x, uint32_t (&kid)[kKids]) {
    uint32_t n = 0;
    if constexpr (W == 0) {
      uint32_t field, count;
      own_slot(t, x, field, count);
      if (count == 0) {
        kid[0] = t.cref == REF_DIRECT ? x + 1 : field;
        kid[1] = t.cref == REF_DIRECT ? x + field : field + 1;
        n = 2;
      }
    } else {
      uint32_t r[W];
      refs(t, x, r);
#pragma unroll
      for (int k = 0; k < W; ++k) {  // interior children to the front
        kid[k] = kEmptyRef;
        if (r[k] != kEmptyRef && ref_is_interior(r[k])) {
#pragma unroll
          for (int j = 0; j <= k; ++j)
            if ((uint32_t)j == n) kid[j] = ref_node(r[k]);
          ++n;
        }
      }
    }
    return n;
  }
  static __device__ __forceinline__ Box3 leaves(const Tree &t, uint32_t x) {
    Box3 b = empty_box();
    if constexpr (W == 0) {
      uint32_t field, count;
      own_slot(t, x, field, count);
      if (count > 0) b = leaf_box(t, field, count);
    } else {
      uint32_t r[W];
      refs(t, x, r);
#pragma unroll
      for (int k = 0; k < W; ++k)
        if (r[k] != kEmptyRef && !ref_is_interior(r[k])) grow(b, leaf_box(t, ref_leaf_first(r[k]), ref_leaf_count(r[k])));
    }
    return b;
  }
};

// ------------------------------------------------------------ kernels
// the vertex table and the direct triangle copies
__global__ void update_kernel(Tree t, const float *__restrict__ v, uint64_t n_verts, uint32_t n_entries) {
  const uint64_t step = (uint64_t)gridDim.x * blockDim.x, i0 = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x;
  for (uint64_t i = i0; i < n_verts; i += step) t.verts[i] = make_float4(v[3 * i], v[3 * i + 1], v[3 * i + 2], 0.f);
  for (uint64_t e = i0; e < n_entries; e += step) {
    float4 *q = t.prims + 3 * e;
    const uint32_t id = __float_as_uint(q[0].w);
    uint32_t i[3];
    triangle_verts(t, id, i);
    for (int k = 0; k < 3; ++k) {
      const float *p = v + 3 * (size_t)i[k];
      q[k] = make_float4(__ldg(p), __ldg(p + 1), __ldg(p + 2), k == 0 ? __uint_as_float(id) : 0.f);
    }
  }
}

// parent of every interior child and the number of interior children
template <int W>
__global__ void links_kernel(Tree t, uint32_t *parent, uint32_t *pending) {
  for (uint32_t x = blockIdx.x * blockDim.x + threadIdx.x; x < t.n_nodes; x += gridDim.x * blockDim.x) {
    uint32_t kid[Family<W>::kKids];
    const uint32_t n = Family<W>::kids(t, x, kid);
#pragma unroll
    for (int k = 0; k < Family<W>::kKids; ++k)
      if ((uint32_t)k < n) parent[kid[k]] = x;
    pending[x] = n;
  }
}

template <int W>
__global__ void leaves_kernel(Tree t, Box3 *boxes) {
  for (uint32_t x = blockIdx.x * blockDim.x + threadIdx.x; x < t.n_nodes; x += gridDim.x * blockDim.x)
    store_box(boxes, x, Family<W>::leaves(t, x));
}

// on entry boxes[x] is the box over x's own leaves
template <int W>
__global__ void climb_kernel(Tree t, const uint32_t *__restrict__ parent, uint32_t *pending, Box3 *boxes) {
  for (uint32_t x = blockIdx.x * blockDim.x + threadIdx.x; x < t.n_nodes; x += gridDim.x * blockDim.x) {
    uint32_t kid[Family<W>::kKids];
    if (Family<W>::kids(t, x, kid) != 0) continue;  // decided from the node, not from the counters
    uint32_t p = parent[x];
    while (p != kNoParent) {
      __threadfence();
      if (atomicSub(pending + p, 1u) != 1u) break;  // not the last child of p
      __threadfence();
      const uint32_t n = Family<W>::kids(t, p, kid);
      pending[p] = n;  // for the next refit
      Box3 b = load_box(boxes, p);
#pragma unroll
      for (int k = 0; k < Family<W>::kKids; ++k)
        if ((uint32_t)k < n) grow(b, load_box(boxes, kid[k]));
      store_box(boxes, p, b);
      p = parent[p];
    }
  }
}

// frame[0..8] grid, [9..11] reciprocal bins, [12..17] the pairs of the
// reciprocal q16 steps
__global__ void frame_kernel(Tree t, const Box3 *boxes, float *frame) {
  if (blockIdx.x != 0 || threadIdx.x != 0) return;
  Box3 r = load_box(boxes, 0);
  if (box_is_empty(r))
    for (int a = 0; a < 3; ++a) r.lo[a] = r.hi[a] = 0.0f;
  const Box3 pr = padded(r);
  if (t.prec == PREC_SLAB) {  // the root's carried box
    for (int a = 0; a < 3; ++a) {
      frame[a] = pr.lo[a];
      frame[3 + a] = pr.hi[a];
    }
    return;
  }
  float bins_inv[3];
  world_frame(t.prec, pr, frame, bins_inv);
  for (int a = 0; a < 3; ++a) {
    frame[9 + a] = bins_inv[a];
    const FPair inv = t.prec == PREC_Q16 ? reciprocal_pair(frame[3 + a]) : FPair{0.0f, 0.0f};
    frame[12 + 2 * a] = inv.hi;
    frame[13 + 2 * a] = inv.lo;
  }
}

__global__ void encode_own_kernel(Tree t, const Box3 *boxes, const float *frame, uint32_t *status) {
  float fr[12];
  FPair inv[3];
  for (int k = 0; k < 12; ++k) fr[k] = frame ? frame[k] : 0.f;
  for (int a = 0; a < 3; ++a) inv[a] = frame ? FPair{frame[12 + 2 * a], frame[13 + 2 * a]} : FPair{0.f, 0.f};
  for (uint32_t x = blockIdx.x * blockDim.x + threadIdx.x; x < t.n_nodes; x += gridDim.x * blockDim.x) {
    uint32_t *p = reinterpret_cast<uint32_t *>(t.nodes + (size_t)x * t.stride);
    if (t.prec == PREC_SLAB) {
      uint32_t kid[2];
      if (Family<0>::kids(t, x, kid) == 2)
        encode_slab_planes(load_box(boxes, kid[0]), load_box(boxes, kid[1]), bin_meta_axis(p[3]),
                           reinterpret_cast<uint8_t *>(p));
      continue;
    }
    uint32_t w[6];
    const bool ok = encode_own_box_fast(t.prec, load_box(boxes, x), fr, fr + 9, inv, w);
    const int n = own_box_words(t.prec);
#pragma unroll
    for (int k = 0; k < 6; ++k)
      if (k < n) p[k] = w[k];
    if (!ok) atomicCAS(status, 0u, (uint32_t)SCION_ERR_BAD_INPUT);
  }
}

// Header and boxes of the nodes, a lane per child, through shared memory (a
// node's part is an odd number of words apart from the next: few bank
// conflicts), then written out by the warp word by word.
template <int W, int PREC>
__global__ void __launch_bounds__(kEncodeThreads) encode_wide_kernel(Tree t, const Box3 *boxes, uint32_t *status) {
  constexpr uint32_t kWords = wide_box_words<W, PREC>(), kPitch = kWords | 1u, kPer = 32 / W;  // nodes per warp
  __shared__ uint32_t stage[kEncodeThreads / 32 * kPer * kPitch];
  const uint32_t lane = threadIdx.x & 31u, k = lane % W, j = lane / W;
  uint32_t *const mine = stage + (threadIdx.x >> 5) * (kPer * kPitch);
  const uint32_t step = gridDim.x * (kEncodeThreads / 32) * kPer;
  for (uint32_t base = (blockIdx.x * (kEncodeThreads / 32) + (threadIdx.x >> 5)) * kPer; base < t.n_nodes; base += step) {
    const uint32_t x = base + j;
    Box3 b = empty_box();
    if (x < t.n_nodes) {
      const uint32_t r = Family<W>::ref(t, x, k);
      if (r != kEmptyRef)
        b = ref_is_interior(r) ? load_box(boxes, ref_node(r)) : leaf_box(t, ref_leaf_first(r), ref_leaf_count(r));
    }
    const int bad = encode_wide_lane<W, PREC>(b, !box_is_empty(b), k, t.soa, reinterpret_cast<uint8_t *>(mine + j * kPitch));
    if (bad) atomicCAS(status, 0u, (uint32_t)SCION_ERR_BAD_INPUT);
    __syncwarp();
    const uint32_t m = min(kPer, t.n_nodes - base);
    for (uint32_t i = lane; i < m * kWords; i += 32) {
      const uint32_t n = i / kWords, w = i % kWords;
      reinterpret_cast<uint32_t *>(t.nodes + (size_t)(base + n) * t.stride)[w] = mine[n * kPitch + w];
    }
    __syncwarp();
  }
}

int grid_for(uint64_t n, int threads) {
  const uint64_t b = (n + threads - 1) / threads;
  return (int)(b == 0 ? 1 : (b < 152ull * 32 ? b : 152ull * 32));
}

template <int W>
cudaError_t refit_family(const Tree &t, const RefitBuffers &b, cudaStream_t s) {
  Box3 *boxes = reinterpret_cast<Box3 *>(b.boxes);
  if (b.first) {
    const cudaError_t e = cudaMemsetAsync(b.parent, 0xFF, (size_t)b.n_nodes * sizeof(uint32_t), s);
    if (e != cudaSuccess) return e;
    links_kernel<W><<<grid_for(b.n_nodes, 256), 256, 0, s>>>(t, b.parent, b.pending);
  }
  leaves_kernel<W><<<grid_for(b.n_nodes, 256), 256, 0, s>>>(t, boxes);
  climb_kernel<W><<<grid_for(b.n_nodes, 256), 256, 0, s>>>(t, b.parent, b.pending, boxes);
  return cudaGetLastError();
}

template <int W>
void encode_wide(const Tree &t, const RefitBuffers &b, cudaStream_t s) {
  const Box3 *boxes = reinterpret_cast<const Box3 *>(b.boxes);
  const int grid = grid_for((uint64_t)b.n_nodes * W, kEncodeThreads);
  switch (t.prec) {
    case PREC_F32: encode_wide_kernel<W, PREC_F32><<<grid, kEncodeThreads, 0, s>>>(t, boxes, b.status); break;
    case PREC_F16: encode_wide_kernel<W, PREC_F16><<<grid, kEncodeThreads, 0, s>>>(t, boxes, b.status); break;
    case PREC_U8: encode_wide_kernel<W, PREC_U8><<<grid, kEncodeThreads, 0, s>>>(t, boxes, b.status); break;
    default: encode_wide_kernel<W, PREC_U16><<<grid, kEncodeThreads, 0, s>>>(t, boxes, b.status); break;
  }
}

}  // namespace

cudaError_t refit_launch(const RefitBuffers &b, const float *d_new_verts, cudaStream_t s) {
  Tree t;
  t.nodes = static_cast<uint8_t *>(b.nodes);
  t.nodes2 = static_cast<const uint8_t *>(b.nodes2);
  t.prims = b.desc.prim_ref ? nullptr : static_cast<float4 *>(b.prims);
  t.prim_ids = b.prim_ids;
  t.verts = static_cast<float4 *>(b.verts4);
  t.tri_idx = b.tri_idx;
  t.n_nodes = b.n_nodes;
  t.stride = b.node_stride;
  t.prec = b.desc.box_prec;
  t.soa = b.desc.box_layout;
  t.cref = b.desc.child_ref;
  const uint32_t entries = t.prims ? b.n_leaf_entries : 0u;
  if (b.n_verts || entries)
    update_kernel<<<grid_for(b.n_verts > entries ? b.n_verts : entries, 256), 256, 0, s>>>(t, d_new_verts, b.n_verts,
                                                                                          entries);
  if (b.n_nodes == 0) return cudaGetLastError();
  const uint32_t W = b.own_box ? 0u : b.desc.width;
  cudaError_t e = W == 0 ? refit_family<0>(t, b, s)
                         : (W == 2 ? refit_family<2>(t, b, s) : (W == 4 ? refit_family<4>(t, b, s) : refit_family<8>(t, b, s)));
  if (e != cudaSuccess) return e;
  const bool grid = prec_has_frame(t.prec);
  if (grid) frame_kernel<<<1, 32, 0, s>>>(t, reinterpret_cast<const Box3 *>(b.boxes), b.frame);
  if (W == 0)
    encode_own_kernel<<<grid_for(b.n_nodes, 256), 256, 0, s>>>(t, reinterpret_cast<const Box3 *>(b.boxes),
                                                               grid ? b.frame : nullptr, b.status);
  else if (W == 2) encode_wide<2>(t, b, s);
  else if (W == 4) encode_wide<4>(t, b, s);
  else encode_wide<8>(t, b, s);
  return cudaGetLastError();
}

}  // namespace scion
