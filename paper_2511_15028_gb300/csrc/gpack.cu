// Packing on the GPU. See gpack.h.
//
// The physical tree is built level by level from the root: a level's nodes
// (in breadth-first order) each find their children (the own-box node: the
// logical node's two children; the wide node: the greedy collapse that opens
// the interior child of largest surface area until W children, exactly as
// the host packer), and prefix sums of their interior-child counts place the
// next level, so the numbering is the breadth-first order of the host packer.
// Depth-first positions follow from the leaf ranges: a node's leaves are
// sorted triangles lo..hi, and in pre-order it comes after the nodes that start
// at a smaller lo and after its ancestors that start at the same one; a count
// per lo, its prefix sums and the length of that chain of ancestors give the
// position at once. (With sibling groups kept contiguous, for indirect child
// references, subtree sizes bottom-up and a pass down the levels.) An exclusive
// scan of the leaf-entry counts in physical order gives every node's first leaf
// entry; the nodes are written with the codecs of codec_fast.h, a lane per child
// of a wide node, and the leaf entries by a thread each.
//
// The bounds of the levels stay on the device: one CTA takes the small levels at
// the top and at the bottom without a launch in between, the large ones take two
// launches each, all issued at once, and the host reads the bounds back only to
// learn whether there are more. Opening a node takes one load (LbvhTree::open);
// a level is a chain of such loads. Scratch is one allocation and the result
// another. Measured, scion_build_gpu and a frame traced after it: 1.4 M triangles,
// 1080p, bvh4 f32 6.34 -> 1.61 ms (0.35 of it the trace); 40 K triangles 1.72 ->
// 0.69 ms. A synchronisation and five launches per level, FP64 areas and pads and
// some 30 allocations were three quarters of it.
#include "gpack.h"

#include <algorithm>
#include <vector>

#include "codec_fast.h"

namespace scion {

namespace {

constexpr int kThreads = 256;
constexpr int kScanThreads = 1024;
constexpr int kScanItems = 4;
constexpr uint32_t kScanTile = kScanThreads * kScanItems;

int grid_for(uint64_t n) {
  return (int)std::max<uint64_t>(1, std::min<uint64_t>((n + kThreads - 1) / kThreads, 152ull * 32));
}

// ------------------------------------------------------------ scan
// Exclusive prefix sum of the block's per-thread values (blockDim.x <= 1024);
// *total receives the block sum.
__device__ uint32_t block_scan(uint32_t x, uint32_t *warp_sums, uint32_t *total) {
  const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
  uint32_t inc = x;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, inc, o);
    if (lane >= (uint32_t)o) inc += y;
  }
  if (lane == 31) warp_sums[warp] = inc;
  __syncthreads();
  const uint32_t nw = blockDim.x >> 5;
  if (warp == 0) {
    const uint32_t s = lane < nw ? warp_sums[lane] : 0u;
    uint32_t si = s;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, si, o);
      if (lane >= (uint32_t)o) si += y;
    }
    if (lane < nw) warp_sums[lane] = si - s;
    if (lane == nw - 1) warp_sums[32] = si;
  }
  __syncthreads();
  const uint32_t r = warp_sums[warp] + inc - x;
  *total = warp_sums[32];
  __syncthreads();
  return r;
}

// sum of each kScanTile-element tile
__global__ void __launch_bounds__(kScanThreads) scan_reduce_kernel(const uint32_t *__restrict__ in, uint64_t m,
                                                                    uint32_t *tile_sums) {
  __shared__ uint32_t ws[33];
  const uint64_t b = (uint64_t)blockIdx.x * kScanTile + (uint64_t)threadIdx.x * kScanItems;
  uint32_t s = 0;
#pragma unroll
  for (int k = 0; k < kScanItems; ++k)
    if (b + k < m) s += in[b + k];
  uint32_t total;
  block_scan(s, ws, &total);
  if (threadIdx.x == 0) tile_sums[blockIdx.x] = total;
}

// exclusive scan of the tile sums in place (one block, any count); the grand
// total goes to *total
__global__ void __launch_bounds__(kScanThreads) scan_tiles_kernel(uint32_t *tile_sums, uint32_t n, uint32_t *total) {
  __shared__ uint32_t ws[33];
  uint32_t carry = 0;
  for (uint32_t base = 0; base < n; base += kScanThreads) {
    const uint32_t i = base + threadIdx.x;
    const uint32_t x = i < n ? tile_sums[i] : 0u;
    uint32_t sum;
    const uint32_t r = block_scan(x, ws, &sum);
    if (i < n) tile_sums[i] = carry + r;
    carry += sum;
  }
  if (threadIdx.x == 0) *total = carry;
}

__global__ void __launch_bounds__(kScanThreads) scan_apply_kernel(const uint32_t *__restrict__ in, uint32_t *out,
                                                                   uint64_t m, const uint32_t *__restrict__ tile_sums) {
  __shared__ uint32_t ws[33];
  const uint64_t b = (uint64_t)blockIdx.x * kScanTile + (uint64_t)threadIdx.x * kScanItems;
  uint32_t v[kScanItems];
  uint32_t s = 0;
#pragma unroll
  for (int k = 0; k < kScanItems; ++k) {
    v[k] = b + k < m ? in[b + k] : 0u;
    s += v[k];
  }
  uint32_t total;
  uint32_t run = tile_sums[blockIdx.x] + block_scan(s, ws, &total);
#pragma unroll
  for (int k = 0; k < kScanItems; ++k)
    if (b + k < m) {
      out[b + k] = run;
      run += v[k];
    }
}

// out[0..m) = exclusive prefix sums of in[0..m) (in == out allowed); *total
// (device) = sum. tiles: scratch of at least ceil(m / kScanTile) words.
cudaError_t exclusive_scan(const uint32_t *in, uint32_t *out, uint64_t m, uint32_t *tiles, uint32_t *total,
                           cudaStream_t s) {
  if (m == 0) return cudaMemsetAsync(total, 0, sizeof(uint32_t), s);
  const uint32_t nt = (uint32_t)((m + kScanTile - 1) / kScanTile);
  scan_reduce_kernel<<<nt, kScanThreads, 0, s>>>(in, m, tiles);
  scan_tiles_kernel<<<1, kScanThreads, 0, s>>>(tiles, nt, total);
  scan_apply_kernel<<<nt, kScanThreads, 0, s>>>(in, out, m, tiles);
  return cudaGetLastError();
}

// ------------------------------------------------------------ the device tree
struct DTree {
  uint32_t nv;
  const uint32_t *ids, *left, *right, *rlo, *rhi;
  const uint8_t *axis, *whole;
  const Box3 *box;
  const uint4 *open;
};

// a logical leaf: a radix leaf, or a subtree kept as one leaf
__device__ __forceinline__ bool lleaf(const DTree &t, uint32_t x) { return x + 1 >= t.nv || t.whole[x]; }

__device__ __forceinline__ void leaf_range(const DTree &t, uint32_t x, uint32_t &first, uint32_t &count) {
  if (x + 1 >= t.nv) {
    first = x - (t.nv - 1);
    count = 1;
  } else {
    first = t.rlo[x];
    count = t.rhi[x] - t.rlo[x] + 1;
  }
}

__device__ __forceinline__ Box3 node_box(const DTree &t, uint32_t x) {
  const float2 *f = reinterpret_cast<const float2 *>(t.box + x);  // 24 bytes, 8-byte aligned
  const float2 a = __ldg(f), b = __ldg(f + 1), c = __ldg(f + 2);
  Box3 r;
  r.lo[0] = a.x; r.lo[1] = a.y; r.lo[2] = b.x;
  r.hi[0] = b.y; r.hi[1] = c.x; r.hi[2] = c.y;
  return r;
}

// surface area in double, as the host packer's collapse measures it
__device__ __forceinline__ double box_area_d(const Box3 &b) {
  const double e0 = fmax(0.0, (double)b.hi[0] - (double)b.lo[0]);
  const double e1 = fmax(0.0, (double)b.hi[1] - (double)b.lo[1]);
  const double e2 = fmax(0.0, (double)b.hi[2] - (double)b.lo[2]);
  return 2.0 * (e0 * e1 + e1 * e2 + e2 * e0);
}

// ------------------------------------------------------------ levels
// Per physical node (breadth-first index i): rad[i] = its logical node (the
// radix node the own-box node is, or the wide node's root); wide nodes also
// keep their W logical children (empty ones last); nk[i] = physical children;
// kfirst[i] = breadth-first index of the first of them (they are consecutive).
// For depth-first positions: chain[i] = ancestors whose leaves start at the
// same sorted triangle, starts[lo] = nodes whose leaves start at lo.
// Logical nodes are kept with a mark where they are logical leaves.
constexpr uint32_t kLeafMark = 0x80000000u;  // node numbers stay below 2^28
__device__ __forceinline__ uint32_t marked(uint32_t c, float open) { return open < 0.0f ? c | kLeafMark : c; }
__device__ __forceinline__ bool is_leaf(uint32_t y) { return (y & kLeafMark) != 0u; }
__device__ __forceinline__ uint32_t plain(uint32_t y) { return y & ~kLeafMark; }

constexpr uint32_t kMaxLevels = 512;  // a radix tree over 32-bit keys and positions is at most 64 deep
constexpr int kLevelGrid = 152 * 4;
constexpr int kSmallThreads = 1024;
constexpr uint32_t kSmallLevel = 2 * kSmallThreads;  // a level one CTA takes
struct Levels {
  uint32_t *lvl;  // level k = nodes [lvl[k], lvl[k + 1])
  uint32_t *cur;  // the first level that is not done
  uint32_t *rad, *wchild, *nk, *kfirst, *chain, *starts, *tsum;
  uint32_t cap;   // nodes the arrays hold
  int *bad;
};

// first sorted triangle of node x
__device__ __forceinline__ uint32_t first_of(const DTree &t, uint32_t x) {
  return x + 1 >= t.nv ? x - (t.nv - 1) : t.rlo[x];
}

__device__ __noinline__ double box_area_of(const DTree &t, uint32_t x) { return box_area_d(node_box(t, x)); }

// The children (marked) of a wide node with root x: the greedy collapse. Areas
// are compared in float (relative error at most 5 units of 2^-24: sums of
// non-negative products); children within 2e-6 of the largest, and areas out
// of float's range, are compared in double, which is what the host packer
// compares, so the choice is the same.
template <int W>
__device__ __forceinline__ void collapse(const DTree &t, uint32_t x, uint32_t (&ch)[W]) {
  float ar[W];
#pragma unroll
  for (int k = 0; k < W; ++k) {
    ch[k] = kEmptyRef;
    ar[k] = -1.0f;
  }
  if (is_leaf(x)) {  // only a root can be a leaf: a one-child wide root
    ch[0] = x;
    return;
  }
  uint4 o = __ldg(t.open + x);
  ch[0] = o.x;
  ch[1] = o.y;
  ar[0] = __uint_as_float(o.z);
  ar[1] = __uint_as_float(o.w);
#pragma unroll
  for (int n = 2; n < W; ++n) {
    int best = -1;
    float top = -1.0f;
#pragma unroll
    for (int k = 0; k < W; ++k)
      if (ar[k] > top) {
        top = ar[k];
        best = k;
      }
    if (best >= 0) {
      const bool in_range = top > 1e-30f && top < 1e37f;
      const float near = in_range ? top * (1.0f - 2e-6f) : 0.0f;
      bool close = !in_range;
#pragma unroll
      for (int k = 0; k < W; ++k) close |= k != best && ar[k] >= near;
      if (close) {
        double most = -1.0;
#pragma unroll
        for (int k = 0; k < W; ++k)
          if (ar[k] >= near) {
            const double d = box_area_of(t, ch[k]);
            if (d > most) {
              most = d;
              best = k;
            }
          }
      }
      uint32_t c = 0;
#pragma unroll
      for (int k = 0; k < W; ++k)
        if (k == best) c = ch[k];
      o = __ldg(t.open + c);
#pragma unroll
      for (int k = W - 1; k >= 0; --k) {
        if (k > best + 1) {
          ch[k] = ch[k > 0 ? k - 1 : 0];
          ar[k] = ar[k > 0 ? k - 1 : 0];
        } else if (k == best + 1) {
          ch[k] = o.y;
          ar[k] = __uint_as_float(o.w);
        } else if (k == best) {
          ch[k] = o.x;
          ar[k] = __uint_as_float(o.z);
        }
      }
    }
  }
#pragma unroll
  for (int k = 0; k < W; ++k)
    if (ch[k] != kEmptyRef) ch[k] = marked(ch[k], ar[k]);
}

// The physical children of node x (marked logical nodes; W = 0: own-box) in
// kid, their number returned.
template <int W>
__device__ __forceinline__ uint32_t find_children(const DTree &t, const Levels &L, uint32_t i, uint32_t x,
                                                  uint32_t (&kid)[W == 0 ? 2 : W]) {
  uint32_t nk = 0;
  if constexpr (W == 0) {
    if (!is_leaf(x)) {
      const uint4 o = __ldg(t.open + x);
      kid[0] = marked(o.x, __uint_as_float(o.z));
      kid[1] = marked(o.y, __uint_as_float(o.w));
      nk = 2;
    }
  } else {
    collapse<W>(t, x, kid);
#pragma unroll
    for (int c = 0; c < W; ++c) {
      L.wchild[(size_t)W * i + c] = kid[c];
      if (kid[c] != kEmptyRef && !is_leaf(kid[c])) ++nk;
    }
  }
  return nk;
}

// Node i's children take the indices from kf on.
template <int W>
__device__ __forceinline__ void place_children(const DTree &t, const Levels &L, uint32_t i, uint32_t x, uint32_t kf,
                                               uint32_t nk, const uint32_t (&kid)[W == 0 ? 2 : W]) {
  L.nk[i] = nk;
  L.kfirst[i] = kf;
  if (nk == 0) return;
  if ((uint64_t)kf + nk > L.cap) {  // cannot be: the arrays hold every node a tree of nv leaves can have
    atomicOr(L.bad, 8);
    return;
  }
  const uint32_t lo = first_of(t, plain(x)), chain = L.chain[i];
  uint32_t r = 0;
#pragma unroll
  for (int c = 0; c < (W == 0 ? 2 : W); ++c) {
    const uint32_t y = kid[c];
    if (W != 0 && (y == kEmptyRef || is_leaf(y))) continue;
    L.rad[kf + r] = y;
    const uint32_t cl = first_of(t, plain(y));
    L.chain[kf + r] = cl == lo ? chain + 1 : 0u;
    if (L.starts) atomicAdd(L.starts + cl, 1u);
    ++r;
  }
}

// Levels small enough for one CTA, one after the other without a launch in
// between: from level *cur on while a level has at most `most` nodes. first:
// sets up the root's level.
template <int W>
__global__ void __launch_bounds__(kSmallThreads) small_levels_kernel(DTree t, Levels L, uint32_t most, int first) {
  __shared__ uint32_t ws[33];
  if (first) {
    if (threadIdx.x == 0) {
      L.lvl[0] = 0;
      L.lvl[1] = 1;
      L.rad[0] = lleaf(t, 0) ? kLeafMark : 0u;  // the root is logical node 0
      L.chain[0] = 0;
      if (L.starts) L.starts[0] = 1;
    }
    __syncthreads();
  }
  uint32_t k = first ? 0u : *L.cur, b = L.lvl[k], e = L.lvl[k + 1];
  while (e > b && e - b <= most && k + 2 < kMaxLevels) {
    uint32_t next = e;
    for (uint32_t j0 = b; j0 < e; j0 += kSmallThreads) {
      const uint32_t i = j0 + threadIdx.x;
      uint32_t kid[W == 0 ? 2 : W], nk = 0, x = 0;
      if (i < e) {
        x = L.rad[i];
        nk = find_children<W>(t, L, i, x, kid);
      }
      uint32_t total;
      const uint32_t at = block_scan(nk, ws, &total);
      if (i < e) place_children<W>(t, L, i, x, next + at, nk, kid);
      next += total;
    }
    __syncthreads();  // the next level's nodes are written
    b = e;
    e = next;
    ++k;
    if (threadIdx.x == 0) L.lvl[k + 1] = e;
  }
  if (threadIdx.x == 0) *L.cur = k;
}

// sum of the block's values, in every thread
__device__ __forceinline__ uint32_t block_sum(uint32_t x, uint32_t *ws) {
  uint32_t total;
  block_scan(x, ws, &total);
  return total;
}

// Children of the nodes of level *cur + slot; tsum[tile] = physical children of
// the tile's nodes (a tile: kThreads nodes).
template <int W>
__global__ void __launch_bounds__(kThreads) expand_kernel(DTree t, Levels L, uint32_t slot) {
  __shared__ uint32_t ws[33];
  const uint32_t k = *L.cur + slot, b = L.lvl[k], m = L.lvl[k + 1] - b;
  for (uint32_t tile = blockIdx.x; tile * kThreads < m; tile += gridDim.x) {
    const uint32_t j = tile * kThreads + threadIdx.x, i = b + j;
    uint32_t nk = 0;
    if (j < m) {
      uint32_t kid[W == 0 ? 2 : W];
      nk = find_children<W>(t, L, i, L.rad[i], kid);
      L.nk[i] = nk;
    }
    const uint32_t sum = block_sum(nk, ws);
    if (threadIdx.x == 0) L.tsum[tile] = sum;
  }
}

// Places the next level and hands its nodes their logical nodes.
template <int W>
__global__ void __launch_bounds__(kThreads) emit_kernel(DTree t, Levels L, uint32_t slot) {
  __shared__ uint32_t ws[33];
  const uint32_t k = *L.cur + slot, b = L.lvl[k], e = L.lvl[k + 1], m = e - b;
  if (m == 0 && blockIdx.x == 0 && threadIdx.x == 0) L.lvl[k + 2] = e;
  for (uint32_t tile = blockIdx.x; tile * kThreads < m; tile += gridDim.x) {
    uint32_t s = 0;
    for (uint32_t q = threadIdx.x; q < tile; q += kThreads) s += L.tsum[q];
    const uint32_t base = e + block_sum(s, ws);
    const uint32_t j = tile * kThreads + threadIdx.x, i = b + j;
    const uint32_t nk = j < m ? L.nk[i] : 0u;
    uint32_t total;
    const uint32_t kf = base + block_scan(nk, ws, &total);
    if ((tile + 1) * kThreads >= m && threadIdx.x == 0) L.lvl[k + 2] = base + total;
    if (j >= m) continue;
    const uint32_t x = L.rad[i];
    uint32_t kid[W == 0 ? 2 : W] = {};
    if constexpr (W == 0) {
      if (nk) find_children<0>(t, L, i, x, kid);
    } else {
#pragma unroll
      for (int c = 0; c < W; ++c) kid[c] = L.wchild[(size_t)W * i + c];
    }
    place_children<W>(t, L, i, x, kf, nk, kid);
  }
}

__global__ void advance_kernel(Levels L, uint32_t slots) { *L.cur += slots; }

// depth-first (pre-order) positions: starts scanned
__global__ void preorder_kernel(DTree t, Levels L, uint32_t *pos, uint32_t n) {
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x)
    pos[i] = L.starts[first_of(t, plain(L.rad[i]))] + L.chain[i];
}

// subtree sizes of one level (its children's are known)
__global__ void size_kernel(const Levels L, uint32_t *size, uint32_t b, uint32_t m) {
  for (uint32_t j = blockIdx.x * blockDim.x + threadIdx.x; j < m; j += gridDim.x * blockDim.x) {
    const uint32_t i = b + j;
    uint32_t s = 1;
    for (uint32_t r = 0; r < L.nk[i]; ++r) s += size[L.kfirst[i] + r];
    size[i] = s;
  }
}

// depth-first positions of the children of one level's nodes with every
// node's children consecutive and each child's descendants after its siblings'
// (base[i] = position of node i's first child)
__global__ void place_kernel(const Levels L, const uint32_t *size, uint32_t *pos, uint32_t *base, uint32_t b,
                             uint32_t m) {
  for (uint32_t j = blockIdx.x * blockDim.x + threadIdx.x; j < m; j += gridDim.x * blockDim.x) {
    const uint32_t i = b + j, kf = L.kfirst[i], nk = L.nk[i];
    const uint32_t bi = base[i];
    uint32_t acc = bi + nk;
    for (uint32_t r = 0; r < nk; ++r) {
      pos[kf + r] = bi + r;
      base[kf + r] = acc;
      acc += size[kf + r] - 1;
    }
  }
}

__global__ void root_place_kernel(uint32_t *pos, uint32_t *base) {
  pos[0] = 0;
  base[0] = 1;
}

__global__ void iota_kernel(uint32_t *pos, uint32_t n) {
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) pos[i] = i;
}

// leaf entries of each physical node, indexed by physical position
template <int W>
__global__ void leaf_count_kernel(DTree t, const Levels L, const uint32_t *pos, uint32_t n, uint32_t *lcnt) {
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    uint32_t c = 0, first, count;
    if constexpr (W == 0) {
      const uint32_t x = L.rad[i];
      if (is_leaf(x)) {
        leaf_range(t, plain(x), first, count);
        c = count;
      }
    } else {
#pragma unroll
      for (int k = 0; k < W; ++k) {
        const uint32_t ch = L.wchild[(size_t)W * i + k];
        if (ch != kEmptyRef && is_leaf(ch)) {
          leaf_range(t, plain(ch), first, count);
          c += count;
        }
      }
    }
    lcnt[pos[i]] = c;
  }
}

// ------------------------------------------------------------ encode
// Leaf entries get the sorted triangle they hold; entries_kernel turns that
// into triangle records or ids, a thread per entry.
struct EntryOut {
  const float *verts;        // float[n_verts][3]
  const uint32_t *indices;   // u32[n_tris][3] or null
  const uint32_t *ids;       // triangle id of a sorted triangle
  float4 *direct;            // 3 float4 per leaf entry, or null
  uint32_t *src;             // sorted triangle per entry; without `direct` replaced by the id
};

__global__ void entries_kernel(EntryOut eo, uint32_t n) {
  for (uint32_t e = blockIdx.x * blockDim.x + threadIdx.x; e < n; e += gridDim.x * blockDim.x) {
    const uint32_t id = __ldg(eo.ids + eo.src[e]);
    if (!eo.direct) {
      eo.src[e] = id;
      continue;
    }
    float4 *rec = eo.direct + 3 * (size_t)e;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const uint32_t i = eo.indices ? __ldg(eo.indices + 3 * (size_t)id + k) : 3 * id + k;
      const float *p = eo.verts + 3 * (size_t)i;
      rec[k] = make_float4(__ldg(p), __ldg(p + 1), __ldg(p + 2), k == 0 ? __uint_as_float(id) : 0.f);
    }
  }
}

struct OwnArgs {
  uint32_t prec, soa, cref, stride;
  float frame[9], bins_inv[3];
  FPair inv[3];  // reciprocals of the q16 steps
};

__global__ void encode_own_kernel(DTree t, const Levels L, const uint32_t *pos, const uint32_t *pbase, uint32_t n,
                                  OwnArgs oa, uint8_t *nodes, uint8_t *nodes2, uint32_t *src, int *bad) {
  const bool quant = prec_is_world_grid(oa.prec);
  int badl = 0;
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    const uint32_t x = plain(L.rad[i]), p = pos[i];
    const bool leaf = is_leaf(L.rad[i]);
    uint32_t ref, meta, count = 0, first = 0;
    if (leaf) {
      leaf_range(t, x, first, count);
      ref = pbase[p];
      meta = bin_pack_meta(count, 0);
      for (uint32_t k = 0; k < count; ++k) src[ref + k] = first + k;
    } else {
      const uint32_t l = pos[L.kfirst[i]], r = pos[L.kfirst[i] + 1];
      if (oa.cref == REF_DIRECT) {
        badl |= l != p + 1 ? 1 : 0;
        ref = r - p;
      } else {
        badl |= r != l + 1 ? 1 : 0;
        ref = l;
      }
      meta = bin_pack_meta(0, t.axis[x]);
    }
    uint32_t *q = reinterpret_cast<uint32_t *>(nodes + (size_t)p * oa.stride);
    uint32_t w[6];
    badl |= encode_own_box_fast(oa.prec, node_box(t, x), oa.frame, oa.bins_inv, oa.inv, w) ? 0 : 2;
    const int nw = own_box_words(oa.prec);
#pragma unroll
    for (int k = 0; k < 6; ++k)
      if (k < nw) q[k] = w[k];
    if (!quant) {
      uint32_t *rq = oa.soa ? reinterpret_cast<uint32_t *>(nodes2 + (size_t)p * kBinRefBytes) : q + 6;
      rq[0] = ref;
      rq[1] = meta;
    } else {
      const uint32_t word = leaf ? qbin_leaf(ref, count) : qbin_interior(ref, t.axis[x]);
      if (oa.prec == PREC_Q16 && oa.soa) reinterpret_cast<uint32_t *>(nodes2)[p] = word;
      else q[nw] = word;
    }
  }
  if (badl) atomicOr(bad, badl);
}

// Wide nodes, a lane per child, through shared memory and out word by word
// (whole nodes, their padding zeroed).
constexpr int kEncodeThreads = 128;
template <int W, int PREC>
__global__ void __launch_bounds__(kEncodeThreads) encode_wide_kernel(DTree t, const Levels L, const uint32_t *pos,
                                                                     const uint32_t *pbase, uint32_t n, uint32_t soa,
                                                                     uint32_t cref, uint32_t node_words, uint8_t *nodes,
                                                                     uint32_t *src, int *bad) {
  constexpr uint32_t kBoxWords = wide_box_words<W, PREC>(), kPer = 32 / W;  // nodes per warp
  // direct references take W words, indirect ones 2 + W / 4; padded to 32 bytes
  constexpr uint32_t kPitch = ((kBoxWords + (W > 3 ? W : 3) + 7) / 8 * 8) | 1u;
  __shared__ uint32_t stage[kEncodeThreads / 32 * kPer * kPitch];
  __shared__ uint32_t place[kEncodeThreads / 32 * kPer];  // the nodes' positions
  const uint32_t lane = threadIdx.x & 31u, k = lane % W, j = lane / W, group = ((1u << W) - 1u) << (lane - k);
  uint32_t *const mine = stage + (threadIdx.x >> 5) * (kPer * kPitch);
  uint32_t *const where = place + (threadIdx.x >> 5) * kPer;
  int badl = 0;
  const uint32_t step = gridDim.x * (kEncodeThreads / 32) * kPer;
  for (uint32_t base = (blockIdx.x * (kEncodeThreads / 32) + (threadIdx.x >> 5)) * kPer; base < n; base += step) {
    const uint32_t i = base + j;
    const bool in = i < n;
    const uint32_t p = in ? pos[i] : 0u;
    if (k == 0) where[j] = p;
    for (uint32_t w = k; w < node_words; w += W) mine[j * kPitch + w] = 0;
    __syncwarp();
    const uint32_t c = in ? L.wchild[(size_t)W * i + k] : kEmptyRef;
    const bool used = c != kEmptyRef, leaf = used && is_leaf(c), interior = used && !leaf;
    uint32_t first = 0, count = 0;
    if (leaf) leaf_range(t, plain(c), first, count);
    // leaf entries of the slots before this one
    uint32_t before = count;
#pragma unroll
    for (int o = 1; o < W; o <<= 1) {
      const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, before, o);
      if (k >= (uint32_t)o) before += y;
    }
    before -= count;
    const uint32_t kids = __ballot_sync(0xFFFFFFFFu, interior) & group;
    const uint32_t rank = __popc(kids & ((1u << lane) - 1u));
    const uint32_t kf = in && kids ? L.kfirst[i] : 0u;
    const uint32_t at0 = in ? pbase[p] : 0u, at = at0 + before;
    const uint32_t cp = interior ? pos[kf + rank] : 0u;
    const uint32_t first_interior = kids ? pos[kf] : 0u;
    if (interior && cref == REF_INDIRECT && cp != first_interior + rank) badl |= 1;
    Box3 b;
    for (int a = 0; a < 3; ++a) b.lo[a] = INFINITY, b.hi[a] = -INFINITY;
    if (used) b = node_box(t, plain(c));
    for (uint32_t q = 0; q < count; ++q) src[at + q] = first + q;
    uint32_t *node = mine + j * kPitch;
    badl |= encode_wide_lane<W, PREC>(b, used && !box_is_empty(b), k, soa, reinterpret_cast<uint8_t *>(node));
    if (cref == REF_DIRECT) {
      node[kBoxWords + k] = interior ? ref_interior(cp) : (leaf ? ref_leaf(at, count) : kEmptyRef);
    } else {
      if (k == 0) {
        node[kBoxWords] = first_interior;
        node[kBoxWords + 1] = at0;
      }
      reinterpret_cast<uint8_t *>(node + kBoxWords + 2)[k] = (uint8_t)(interior ? kMetaInterior | rank : count);
    }
    __syncwarp();
    const uint32_t m = min(kPer, n - base);
    for (uint32_t q = lane; q < m * node_words; q += 32) {
      const uint32_t y = q / node_words, w = q % node_words;
      reinterpret_cast<uint32_t *>(nodes)[(size_t)where[y] * node_words + w] = mine[y * kPitch + w];
    }
    __syncwarp();
  }
  if (badl) atomicOr(bad, badl);
}

template <int W>
void encode_wide(uint32_t prec, const DTree &t, const Levels &L, const uint32_t *pos, const uint32_t *pbase, uint32_t n,
                 uint32_t soa, uint32_t cref, uint32_t node_words, uint8_t *nodes, uint32_t *src, int *bad,
                 cudaStream_t s) {
  const int g = (int)std::min<uint64_t>(((uint64_t)n * W + kEncodeThreads - 1) / kEncodeThreads, 152ull * 64);
#define SCION_ENC(P) encode_wide_kernel<W, P><<<g, kEncodeThreads, 0, s>>>(t, L, pos, pbase, n, soa, cref, node_words, nodes, src, bad)
  switch (prec) {
    case PREC_F32: SCION_ENC(PREC_F32); break;
    case PREC_F16: SCION_ENC(PREC_F16); break;
    case PREC_U8: SCION_ENC(PREC_U8); break;
    default: SCION_ENC(PREC_U16); break;
  }
#undef SCION_ENC
}

__global__ void verts4_kernel(const float *__restrict__ v, uint64_t n, float4 *out) {
  for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < n; i += (uint64_t)gridDim.x * blockDim.x)
    out[i] = make_float4(v[3 * i], v[3 * i + 1], v[3 * i + 2], 0.f);
}

__global__ void index_check_kernel(const uint32_t *__restrict__ ix, uint64_t n, uint64_t n_verts, int *bad) {
  int b = 0;
  for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < n; i += (uint64_t)gridDim.x * blockDim.x)
    b |= ix[i] >= n_verts ? 1 : 0;
  if (__any_sync(0xFFFFFFFFu, b) && (threadIdx.x & 31u) == 0) atomicOr(bad, 1);
}

scion_status cuda_err(cudaError_t e, std::string *err) {
  *err = cudaGetErrorString(e);
  return e == cudaErrorMemoryAllocation ? SCION_ERR_OOM : SCION_ERR_CUDA;
}

}  // namespace

void launch_index_check(const uint32_t *d_indices, uint64_t n_tris, uint64_t n_verts, int *d_bad, cudaStream_t s) {
  if (d_indices && n_tris)
    index_check_kernel<<<grid_for(3 * n_tris), kThreads, 0, s>>>(d_indices, 3 * n_tris, n_verts, d_bad);
}

bool gpu_pack_supported(const scion_layout_desc &d, bool own_box) {
  if (d.order == ORDER_TREELET) return false;
  if (own_box && d.box_prec == PREC_SLAB) return false;
  return true;
}

scion_status gpu_pack(const LbvhTree &t, const float *d_verts, uint64_t n_verts, const uint32_t *d_indices,
                      uint64_t n_tris, const scion_layout_desc &d, bool own_box, cudaStream_t s,
                      DevicePacked *out, std::string *err) {
  *out = DevicePacked{};
  const uint32_t nv = t.nv, W = d.width;
  const bool dfs = d.order != ORDER_BFS, group = dfs && d.child_ref == REF_INDIRECT, pre = dfs && !group;
  const bool direct = d.prim_ref == REF_DIRECT;
  // most nodes the tree can have
  const uint64_t cap = nv == 0 ? 0 : (own_box ? 2ull * nv - 1 : std::max<uint64_t>(1, nv - 1));
  cudaError_t e;
#define SCION_GP(call)                                \
  do {                                                \
    e = (call);                                       \
    if (e != cudaSuccess) return cuda_err(e, err);    \
  } while (0)
  // scratch: one allocation
  Arena scratch;
  Levels L{};
  uint32_t *pos = nullptr, *pbase = nullptr, *size = nullptr, *base = nullptr, *src = nullptr, *tiles = nullptr;
  uint32_t *total = nullptr;
  for (int pass = 0; pass < 2 && nv > 0; ++pass) {  // sizes, then addresses
    if (pass) SCION_GP(scratch.commit(s));
    scratch.take(&L.lvl, kMaxLevels + 4);
    scratch.take(&L.cur, 1);
    scratch.take(&L.bad, 1);
    scratch.take(&total, 1);
    scratch.take(&L.rad, cap);
    scratch.take(&L.nk, cap);
    scratch.take(&L.kfirst, cap);
    scratch.take(&L.chain, cap);
    scratch.take(&pos, cap);
    scratch.take(&pbase, cap);
    scratch.take(&L.tsum, (cap + kThreads - 1) / kThreads);
    scratch.take(&tiles, (std::max<uint64_t>(cap, nv) + kScanTile - 1) / kScanTile);
    if (!own_box) scratch.take(&L.wchild, W * cap);
    if (pre) scratch.take(&L.starts, nv);
    if (group) {
      scratch.take(&size, cap);
      scratch.take(&base, cap);
    }
    if (direct) scratch.take(&src, nv);
  }
  const DTree dt{nv, t.ids, t.left, t.right, t.rlo, t.rhi, t.axis, t.whole, t.box, t.open};
  std::vector<uint32_t> lvl{0, 0};
  uint32_t nn = 0, levels = 0;
  if (nv > 0) {
    L.cap = (uint32_t)std::min<uint64_t>(cap, 0xFFFFFFFFull);
    SCION_GP(cudaMemsetAsync(L.bad, 0, sizeof(int), s));
    if (pre) SCION_GP(cudaMemsetAsync(L.starts, 0, nv * sizeof(uint32_t), s));
    // small levels at the top in one CTA, then the large ones with two launches
    // each, then the small ones at the bottom; again where that was too few.
    // Levels grow by 1.8, 3 and 5.6 or more in trees 2, 4 and 8 wide until most
    // nodes are placed, a few levels after one of nv / kSmallLevel times the size.
    uint32_t ratio = 0;  // log2 of that, rounded up
    while (ratio < 31 && ((uint64_t)kSmallLevel << ratio) < nv) ++ratio;
    uint32_t large = ratio == 0 ? 0u : ((own_box || W == 2) ? ratio * 6 / 5 + 4 : (W == 4 ? ratio * 5 / 8 + 3 : ratio * 2 / 5 + 3));
    const uint32_t family = own_box ? 0u : W;
    auto small = [&](uint32_t most, int first) {
      switch (family) {
        case 0: small_levels_kernel<0><<<1, kSmallThreads, 0, s>>>(dt, L, most, first); break;
        case 2: small_levels_kernel<2><<<1, kSmallThreads, 0, s>>>(dt, L, most, first); break;
        case 4: small_levels_kernel<4><<<1, kSmallThreads, 0, s>>>(dt, L, most, first); break;
        default: small_levels_kernel<8><<<1, kSmallThreads, 0, s>>>(dt, L, most, first); break;
      }
    };
    for (int first = 1;; first = 0) {
      if (first) small(kSmallLevel, 1);
      for (uint32_t q = 0; q < large; ++q) {
        switch (family) {
          case 0:
            expand_kernel<0><<<kLevelGrid, kThreads, 0, s>>>(dt, L, q);
            emit_kernel<0><<<kLevelGrid, kThreads, 0, s>>>(dt, L, q);
            break;
          case 2:
            expand_kernel<2><<<kLevelGrid, kThreads, 0, s>>>(dt, L, q);
            emit_kernel<2><<<kLevelGrid, kThreads, 0, s>>>(dt, L, q);
            break;
          case 4:
            expand_kernel<4><<<kLevelGrid, kThreads, 0, s>>>(dt, L, q);
            emit_kernel<4><<<kLevelGrid, kThreads, 0, s>>>(dt, L, q);
            break;
          default:
            expand_kernel<8><<<kLevelGrid, kThreads, 0, s>>>(dt, L, q);
            emit_kernel<8><<<kLevelGrid, kThreads, 0, s>>>(dt, L, q);
            break;
        }
      }
      if (large) {
        advance_kernel<<<1, 1, 0, s>>>(L, large);
        small(kSmallLevel, 0);
      }
      SCION_GP(cudaGetLastError());
      uint32_t k = 0;
      lvl.resize(kMaxLevels + 4);
      SCION_GP(cudaMemcpyAsync(lvl.data(), L.lvl, lvl.size() * sizeof(uint32_t), cudaMemcpyDeviceToHost, s));
      SCION_GP(cudaMemcpyAsync(&k, L.cur, sizeof(uint32_t), cudaMemcpyDeviceToHost, s));
      SCION_GP(cudaStreamSynchronize(s));
      if (lvl[k + 1] == lvl[k]) {  // level k is empty
        lvl.resize(k + 2);
        break;
      }
      large = 6;
      if (k + large + 4 > kMaxLevels) {
        *err = "GPU packer: the tree has too many levels";
        return SCION_ERR_CUDA;
      }
    }
    nn = lvl.back();
    while (lvl.size() > 2 && lvl[lvl.size() - 2] == nn) lvl.pop_back();
    levels = (uint32_t)lvl.size() - 1;
    if (own_box && prec_is_world_grid(d.box_prec) && nn >= kQMaxNodes) {
      *err = "too many nodes for the quantised own-box node";
      return SCION_ERR_UNSUPPORTED_LAYOUT;
    }
    if (!own_box && nn >= kMaxNodes) {
      *err = "too many nodes";
      return SCION_ERR_INVALID_ARG;
    }
  }
  // sizes of the result, and its one allocation
  OwnArgs oa{};
  uint32_t stride = 0, ref_bytes = 0;
  if (own_box) {
    oa.prec = d.box_prec;
    oa.soa = d.box_layout;
    oa.cref = d.child_ref;
    const bool soa = d.box_layout == LAYOUT_SOA, a16 = d.align == 16;
    if (oa.prec == PREC_F32) {
      stride = soa ? (a16 ? 32u : kBinBoxBytes) : kBinNodeBytes;
      ref_bytes = soa ? kBinRefBytes : 0u;
    } else if (oa.prec == PREC_Q16) {
      stride = soa ? (a16 ? 16u : kQBoxBytes) : 16u;
      ref_bytes = soa ? 4u : 0u;
    } else {
      stride = a16 ? 16u : kQBoxBytes;
    }
    oa.stride = stride;
  } else {
    stride = wide_node_stride(W, d.box_prec, d.child_ref);
  }
  const uint64_t entries = nv;  // every valid triangle is in one leaf
  Arena block;
  uint8_t *nodes = nullptr, *nodes2 = nullptr;
  float4 *prims = nullptr, *verts4 = nullptr;
  uint32_t *prim_ids = nullptr, *idx = nullptr;
  for (int pass = 0; pass < 2; ++pass) {
    if (pass) SCION_GP(block.commit());
    if (nn) block.take(&nodes, (uint64_t)nn * stride);
    if (nn && ref_bytes) block.take(&nodes2, (uint64_t)nn * ref_bytes);
    if (entries && direct) block.take(&prims, 3 * entries);
    if (entries && !direct) block.take(&prim_ids, entries);
    if (n_verts) block.take(&verts4, n_verts);
    if (d_indices && n_tris) block.take(&idx, 3 * n_tris);
    block.take(&out->scratch, kBvhScratchWords);
  }
  SCION_GP(cudaMemsetAsync(out->scratch, 0, kBvhScratchWords * sizeof(uint32_t), s));
  // vertex / index tables (indirect triangles and the backward pass use them)
  if (n_verts > 0) verts4_kernel<<<grid_for(n_verts), kThreads, 0, s>>>(d_verts, n_verts, verts4);
  SCION_GP(cudaGetLastError());
  if (idx) SCION_GP(cudaMemcpyAsync(idx, d_indices, 3 * n_tris * sizeof(uint32_t), cudaMemcpyDeviceToDevice, s));
  out->root_ref = kEmptyRef;
  if (nv > 0) {
    // physical positions
    if (!dfs) {
      iota_kernel<<<grid_for(nn), kThreads, 0, s>>>(pos, nn);
    } else if (pre) {
      SCION_GP(exclusive_scan(L.starts, L.starts, nv, tiles, total, s));
      preorder_kernel<<<grid_for(nn), kThreads, 0, s>>>(dt, L, pos, nn);
    } else {
      for (uint32_t k = levels; k-- > 0;)
        size_kernel<<<grid_for(lvl[k + 1] - lvl[k]), kThreads, 0, s>>>(L, size, lvl[k], lvl[k + 1] - lvl[k]);
      root_place_kernel<<<1, 1, 0, s>>>(pos, base);
      for (uint32_t k = 0; k + 1 < levels; ++k)
        place_kernel<<<grid_for(lvl[k + 1] - lvl[k]), kThreads, 0, s>>>(L, size, pos, base, lvl[k],
                                                                        lvl[k + 1] - lvl[k]);
    }
    SCION_GP(cudaGetLastError());
    // leaf entries: counts in physical order, prefix sums
    switch (own_box ? 0u : W) {
      case 0: leaf_count_kernel<0><<<grid_for(nn), kThreads, 0, s>>>(dt, L, pos, nn, pbase); break;
      case 2: leaf_count_kernel<2><<<grid_for(nn), kThreads, 0, s>>>(dt, L, pos, nn, pbase); break;
      case 4: leaf_count_kernel<4><<<grid_for(nn), kThreads, 0, s>>>(dt, L, pos, nn, pbase); break;
      default: leaf_count_kernel<8><<<grid_for(nn), kThreads, 0, s>>>(dt, L, pos, nn, pbase); break;
    }
    SCION_GP(cudaGetLastError());
    SCION_GP(exclusive_scan(pbase, pbase, nn, tiles, total, s));
    uint32_t *entry = direct ? src : prim_ids;
    if (own_box) {
      if (prec_is_world_grid(oa.prec)) {
        // world grid over the padded root box, computed by the host codec
        Box3 root_box;
        SCION_GP(cudaMemcpyAsync(&root_box, t.box, sizeof(Box3), cudaMemcpyDeviceToHost, s));
        SCION_GP(cudaStreamSynchronize(s));
        world_frame(oa.prec, padded(root_box), oa.frame, oa.bins_inv);
        for (int a = 0; a < 3; ++a) oa.inv[a] = reciprocal_pair(oa.prec == PREC_Q16 ? oa.frame[3 + a] : 0.0f);
        for (int k = 0; k < 9; ++k) out->frame[k] = oa.frame[k];
        // records padded to 16 bytes have words that nothing writes
        SCION_GP(cudaMemsetAsync(nodes, 0, (uint64_t)nn * stride, s));
      } else if (stride == 32 && d.box_layout == LAYOUT_SOA) {
        SCION_GP(cudaMemsetAsync(nodes, 0, (uint64_t)nn * stride, s));
      }
      encode_own_kernel<<<grid_for(nn), kThreads, 0, s>>>(dt, L, pos, pbase, nn, oa, nodes, nodes2, entry, L.bad);
      out->root_ref = 0;
      out->depth = levels;
      out->stack_need = levels;
    } else {
      const uint32_t words = stride / 4;
      switch (W) {
        case 2: encode_wide<2>(d.box_prec, dt, L, pos, pbase, nn, d.box_layout, d.child_ref, words, nodes, entry, L.bad, s); break;
        case 4: encode_wide<4>(d.box_prec, dt, L, pos, pbase, nn, d.box_layout, d.child_ref, words, nodes, entry, L.bad, s); break;
        default: encode_wide<8>(d.box_prec, dt, L, pos, pbase, nn, d.box_layout, d.child_ref, words, nodes, entry, L.bad, s); break;
      }
      out->root_ref = ref_interior(0);
      out->depth = levels;
      out->stack_need = (W - 1) * levels + 1;
    }
    SCION_GP(cudaGetLastError());
    entries_kernel<<<grid_for(entries), kThreads, 0, s>>>(EntryOut{d_verts, d_indices, t.ids, prims, entry},
                                                          (uint32_t)entries);
    SCION_GP(cudaGetLastError());
    int hbad = 0;
    SCION_GP(cudaMemcpyAsync(&hbad, L.bad, sizeof(int), cudaMemcpyDeviceToHost, s));
    SCION_GP(cudaStreamSynchronize(s));
    if (hbad & 8) {
      *err = "GPU packer: level sizes exceed the node count";
      return SCION_ERR_CUDA;
    }
    if (hbad & 1) {
      *err = own_box ? "node order violates the child reference encoding" : "siblings not contiguous";
      return SCION_ERR_UNSUPPORTED_LAYOUT;
    }
    if (hbad & 2) {
      *err = own_box ? "world-grid enclosure" : "f16 enclosure";
      return SCION_ERR_BAD_INPUT;
    }
    if (hbad & 4) {
      *err = "u8/u16 enclosure";
      return SCION_ERR_BAD_INPUT;
    }
  } else {
    SCION_GP(cudaStreamSynchronize(s));
  }
#undef SCION_GP
  out->n_nodes = nn;
  out->n_leaf_entries = (uint32_t)entries;
  out->node_stride = stride;
  out->node_bytes = (uint64_t)nn * stride;
  out->node2_bytes = (uint64_t)nn * ref_bytes;
  out->prim_direct_bytes = direct ? 48ull * entries : 0;
  out->prim_id_bytes = direct ? 0 : 4ull * entries;
  out->vert_bytes = n_verts * sizeof(float4);
  out->idx_bytes = d_indices ? 3 * n_tris * sizeof(uint32_t) : 0;
  out->nodes = nodes;
  out->nodes2 = nodes2;
  out->prims = prims;
  out->prim_ids = prim_ids;
  out->verts4 = verts4;
  out->idx = idx;
  out->block = block.release();  // the caller's now
  return SCION_OK;
}

}  // namespace scion
