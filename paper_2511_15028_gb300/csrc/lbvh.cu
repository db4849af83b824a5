// Linear BVH construction on the GPU. See lbvh.h.
//
// Steps, each its own kernel on the caller's stream:
//   1. triangle boxes, centroid bounds (ordered-integer atomics), valid count;
//   2. 30-bit Morton code of each centroid (10 bits per axis, x highest);
//      triangles with a non-finite vertex get the code 0xFFFFFFFF;
//   3. stable LSD radix sort of (code, triangle) pairs, 8-bit digits, 4
//      passes; each pass = per-tile digit histogram, an exclusive scan along
//      each digit's tiles (a CTA per digit), and a scatter in which each warp
//      ranks its keys with match votes and the tile is put in digit order in
//      shared memory first, so that it leaves in runs. (4-bit digits took
//      twice the passes over the pairs, each with a scan by one CTA.)
//   4. binary radix tree over the sorted codes, one thread per interior node
//      (Karras 2012, "Maximizing parallelism in the construction of BVHs,
//      octrees, and k-d trees"); equal codes are ordered by their position;
//   5. boxes bottom-up: a thread per leaf climbs while it is the second of
//      the two children to arrive at a node (an atomic counter per node;
//      nothing waits on another thread), and on the way the leaf choice: a
//      subtree of at most leaf_max triangles becomes one leaf where the
//      surface area heuristic prefers it to the subtree's best split. Costs
//      are only computed for such subtrees (no larger one can become a leaf),
//      in FP32 with an error bound; what that cannot decide is decided in
//      double.
// Measured for 1.4 M triangles (ncu, kernels alone): bounds 96 -> 14 us (seven
// atomics per CTA instead of per warp), sort 283 -> 104, boxes and leaf choice
// 274 + 832 -> 192 (the costs were in FP64 for every node, and both climbs went
// through L2 from the leaves up). The boxes' least traffic is 0.17 GB, 25 us; the
// climb above the tiles is a chain of dependent L2 round trips.
#include "lbvh.h"

#include "gpack.h"

#include <algorithm>
#include <cmath>
#include <cstring>
#include <mutex>
#include <vector>

namespace scion {

namespace {

constexpr uint32_t kInvalidKey = 0xFFFFFFFFu;
constexpr uint32_t kNone = 0xFFFFFFFFu;
constexpr int kSortThreads = 256;
constexpr int kSortItems = 16;
constexpr int kSortTile = kSortThreads * kSortItems;  // keys per sort tile
constexpr int kRadix = 256;                            // 8-bit digits
constexpr int kSortWarps = kSortThreads / 32;

// order-preserving float <-> u32 map (for atomicMin / atomicMax on floats)
__device__ __forceinline__ uint32_t f2o(float f) {
  const uint32_t u = __float_as_uint(f);
  return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}
__device__ __forceinline__ float o2f(uint32_t u) {
  return __uint_as_float((u & 0x80000000u) ? (u & 0x7FFFFFFFu) : ~u);
}

__device__ __forceinline__ bool finite3(float a, float b, float c) {
  return isfinite(a) && isfinite(b) && isfinite(c);
}

// a box as three 8-byte words (boxes are 24 bytes, 8-byte aligned)
__device__ __forceinline__ void store_box(Box3 *p, const Box3 &b) {
  float2 *f = reinterpret_cast<float2 *>(p);
  f[0] = make_float2(b.lo[0], b.lo[1]);
  f[1] = make_float2(b.lo[2], b.hi[0]);
  f[2] = make_float2(b.hi[1], b.hi[2]);
}
__device__ __forceinline__ Box3 unpack_box(float2 a, float2 b, float2 c) {
  Box3 r;
  r.lo[0] = a.x; r.lo[1] = a.y; r.lo[2] = b.x;
  r.hi[0] = b.y; r.hi[1] = c.x; r.hi[2] = c.y;
  return r;
}
// read past L1: other SMs write the boxes in the same launch
__device__ __forceinline__ Box3 load_box_l2(const Box3 *p) {
  const float2 *f = reinterpret_cast<const float2 *>(p);
  return unpack_box(__ldcg(f), __ldcg(f + 1), __ldcg(f + 2));
}

// 1. triangle boxes (empty when not finite), centroid bounds cb[0..2] min,
//    cb[3..5] max (ordered u32), valid count; one set of atomics per CTA
constexpr int kBoundsThreads = 256;
__global__ void __launch_bounds__(kBoundsThreads) tri_bounds_kernel(const float *__restrict__ v,
                                                                    const uint32_t *__restrict__ ix, uint32_t n,
                                                                    Box3 *__restrict__ tbox, uint32_t *cb,
                                                                    uint32_t *n_valid, const int *bad_index) {
  __shared__ uint32_t part[7][kBoundsThreads / 32];
  if (*bad_index) return;  // nothing is read through indices out of range
  uint32_t mn[3] = {0xFFFFFFFFu, 0xFFFFFFFFu, 0xFFFFFFFFu}, mx[3] = {0u, 0u, 0u};
  uint32_t cnt = 0;
  for (uint32_t t = blockIdx.x * blockDim.x + threadIdx.x; t < n; t += gridDim.x * blockDim.x) {
    const uint32_t i0 = ix ? ix[3 * (size_t)t] : 3 * t;
    const uint32_t i1 = ix ? ix[3 * (size_t)t + 1] : 3 * t + 1;
    const uint32_t i2 = ix ? ix[3 * (size_t)t + 2] : 3 * t + 2;
    const float *p0 = v + 3 * (size_t)i0, *p1 = v + 3 * (size_t)i1, *p2 = v + 3 * (size_t)i2;
    const bool ok = finite3(p0[0], p0[1], p0[2]) && finite3(p1[0], p1[1], p1[2]) && finite3(p2[0], p2[1], p2[2]);
    Box3 b;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      b.lo[a] = fminf(fminf(p0[a], p1[a]), p2[a]);
      b.hi[a] = fmaxf(fmaxf(p0[a], p1[a]), p2[a]);
      if (!ok) {
        b.lo[a] = __int_as_float(0x7f800000);
        b.hi[a] = -__int_as_float(0x7f800000);
      } else {
        const uint32_t c = f2o((p0[a] + p1[a] + p2[a]) * (1.0f / 3.0f));
        mn[a] = min(mn[a], c);
        mx[a] = max(mx[a], c);
      }
    }
    store_box(tbox + t, b);
    cnt += ok ? 1u : 0u;
  }
  const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const uint32_t x = __reduce_min_sync(0xFFFFFFFFu, mn[a]), y = __reduce_max_sync(0xFFFFFFFFu, mx[a]);
    if (lane == 0) {
      part[a][warp] = x;
      part[3 + a][warp] = y;
    }
  }
  cnt = __reduce_add_sync(0xFFFFFFFFu, cnt);
  if (lane == 0) part[6][warp] = cnt;
  __syncthreads();
  if (threadIdx.x < 7) {
    uint32_t x = part[threadIdx.x][0];
    for (int w = 1; w < kBoundsThreads / 32; ++w) {
      const uint32_t y = part[threadIdx.x][w];
      x = threadIdx.x < 3 ? min(x, y) : (threadIdx.x < 6 ? max(x, y) : x + y);
    }
    if (threadIdx.x < 3) atomicMin(cb + threadIdx.x, x);
    else if (threadIdx.x < 6) atomicMax(cb + threadIdx.x, x);
    else atomicAdd(n_valid, x);
  }
}

// spread the low 10 bits of x to every third bit
__device__ __forceinline__ uint32_t spread3(uint32_t x) {
  x &= 0x3FFu;
  x = (x | (x << 16)) & 0x030000FFu;
  x = (x | (x << 8)) & 0x0300F00Fu;
  x = (x | (x << 4)) & 0x030C30C3u;
  x = (x | (x << 2)) & 0x09249249u;
  return x;
}

// 2. Morton codes of the triangle centroids (same centroid as the bounds pass)
__global__ void morton_kernel(const float *__restrict__ v, const uint32_t *__restrict__ ix,
                              const Box3 *__restrict__ tbox, uint32_t n, const uint32_t *cb, uint32_t *keys,
                              uint32_t *vals, const int *bad_index) {
  if (*bad_index) return;
  float lo[3], sc[3];
  for (int a = 0; a < 3; ++a) {
    lo[a] = o2f(cb[a]);
    const float ext = o2f(cb[3 + a]) - lo[a];
    sc[a] = ext > 0.0f ? 1024.0f / ext : 0.0f;
  }
  for (uint32_t t = blockIdx.x * blockDim.x + threadIdx.x; t < n; t += gridDim.x * blockDim.x) {
    uint32_t key = kInvalidKey;
    if (tbox[t].lo[0] <= tbox[t].hi[0]) {
      const uint32_t i0 = ix ? ix[3 * (size_t)t] : 3 * t;
      const uint32_t i1 = ix ? ix[3 * (size_t)t + 1] : 3 * t + 1;
      const uint32_t i2 = ix ? ix[3 * (size_t)t + 2] : 3 * t + 2;
      uint32_t q[3];
      for (int a = 0; a < 3; ++a) {
        const float c = (v[3 * (size_t)i0 + a] + v[3 * (size_t)i1 + a] + v[3 * (size_t)i2 + a]) * (1.0f / 3.0f);
        const float f = (c - lo[a]) * sc[a];
        q[a] = f >= 1023.0f ? 1023u : (f > 0.0f ? (uint32_t)f : 0u);
      }
      key = (spread3(q[0]) << 2) | (spread3(q[1]) << 1) | spread3(q[2]);
    }
    keys[t] = key;
    vals[t] = t;
  }
}

// 3a. digit histogram of one tile of kSortTile keys: hist[digit * tiles + tile]
__global__ void __launch_bounds__(kSortThreads) radix_hist_kernel(const uint32_t *__restrict__ keys, int shift,
                                                                   uint32_t *hist, uint32_t tiles) {
  __shared__ uint32_t cnt[kRadix];
  cnt[threadIdx.x] = 0;  // kSortThreads == kRadix
  __syncthreads();
  const uint4 *p = reinterpret_cast<const uint4 *>(keys + (size_t)blockIdx.x * kSortTile);
#pragma unroll
  for (int i = 0; i < kSortItems / 4; ++i) {
    const uint4 k = p[i * kSortThreads + threadIdx.x];
    atomicAdd(&cnt[(k.x >> shift) & 255u], 1u);
    atomicAdd(&cnt[(k.y >> shift) & 255u], 1u);
    atomicAdd(&cnt[(k.z >> shift) & 255u], 1u);
    atomicAdd(&cnt[(k.w >> shift) & 255u], 1u);
  }
  __syncthreads();
  hist[(size_t)threadIdx.x * tiles + blockIdx.x] = cnt[threadIdx.x];
}

// Exclusive prefix sum of the 256 per-thread values of a block (returns the
// thread's prefix; *total receives the block sum).
__device__ __forceinline__ uint32_t block_exclusive_scan(uint32_t x, uint32_t *warp_sums, uint32_t *total) {
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
    uint32_t s = lane < nw ? warp_sums[lane] : 0u;
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

// 3b. exclusive scan of one digit's tiles in place; totals[digit] = their sum
__global__ void __launch_bounds__(kSortThreads) radix_scan_kernel(uint32_t *hist, uint32_t tiles, uint32_t *totals) {
  __shared__ uint32_t warp_sums[33];
  uint32_t *row = hist + (size_t)blockIdx.x * tiles;
  uint32_t carry = 0;
  for (uint32_t b = 0; b < tiles; b += kSortThreads) {
    const uint32_t i = b + threadIdx.x;
    const uint32_t x = i < tiles ? row[i] : 0u;
    uint32_t sum;
    const uint32_t r = block_exclusive_scan(x, warp_sums, &sum);
    if (i < tiles) row[i] = carry + r;
    carry += sum;
  }
  if (threadIdx.x == 0) totals[blockIdx.x] = carry;
}

// Place of a lane's key among its warp's keys of digit d so far, in lane order;
// counts them.
__device__ __forceinline__ uint32_t rank_in_warp(uint32_t *cnt, uint32_t d, uint32_t lane) {
  const uint32_t peers = __match_any_sync(0xFFFFFFFFu, d);
  const uint32_t before = __popc(peers & ((1u << lane) - 1u));
  const uint32_t seen = cnt[d];
  __syncwarp();
  if (before == 0) cnt[d] = seen + __popc(peers);
  __syncwarp();
  return seen + before;
}

// 3c. stable scatter of one tile. Warp w holds keys w*512 .. w*512+511, item i
// of a lane being key i*32 + lane of them.
__global__ void __launch_bounds__(kSortThreads) radix_scatter_kernel(const uint32_t *__restrict__ kin,
                                                                      const uint32_t *__restrict__ vin,
                                                                      uint32_t *__restrict__ kout,
                                                                      uint32_t *__restrict__ vout, int shift,
                                                                      const uint32_t *__restrict__ hist,
                                                                      const uint32_t *__restrict__ totals,
                                                                      uint32_t tiles) {
  __shared__ uint32_t cnt[kSortWarps][kRadix];  // per warp: keys of each digit so far
  __shared__ uint32_t start[kRadix];            // first place of a digit within the tile
  __shared__ uint32_t dest[kRadix];             // global place of a digit's first key, less `start`
  __shared__ uint32_t buf[kSortTile];           // the tile in digit order, keys then triangles
  __shared__ uint32_t warp_sums[33];
  const uint32_t t = threadIdx.x, lane = t & 31u, warp = t >> 5;
  const size_t base = (size_t)blockIdx.x * kSortTile + (size_t)warp * (32 * kSortItems) + lane;
  for (int i = t; i < kSortWarps * kRadix; i += kSortThreads) (&cnt[0][0])[i] = 0;
  __syncthreads();
  uint32_t k[kSortItems], val[kSortItems], place[kSortItems];
#pragma unroll
  for (int i = 0; i < kSortItems; ++i) {
    k[i] = kin[base + 32 * i];
    val[i] = vin[base + 32 * i];
  }
#pragma unroll
  for (int i = 0; i < kSortItems; ++i) place[i] = rank_in_warp(cnt[warp], (k[i] >> shift) & 255u, lane);
  __syncthreads();
  // digit t (kSortThreads == kRadix): its warps in order, its place in the
  // tile and in the output
  uint32_t run = 0;
#pragma unroll
  for (int w = 0; w < kSortWarps; ++w) {
    const uint32_t x = cnt[w][t];
    cnt[w][t] = run;
    run += x;
  }
  uint32_t total;
  const uint32_t in_tile = block_exclusive_scan(run, warp_sums, &total);
  const uint32_t digit_base = block_exclusive_scan(totals[t], warp_sums, &total);
  start[t] = in_tile;
  dest[t] = digit_base + hist[(size_t)t * tiles + blockIdx.x] - in_tile;
  __syncthreads();
#pragma unroll
  for (int i = 0; i < kSortItems; ++i) {
    const uint32_t d = (k[i] >> shift) & 255u;
    place[i] += start[d] + cnt[warp][d];
    buf[place[i]] = k[i];
  }
  __syncthreads();
  uint32_t out[kSortItems];
#pragma unroll
  for (int i = 0; i < kSortItems; ++i) {
    const uint32_t j = i * kSortThreads + t, key = buf[j];
    out[i] = dest[(key >> shift) & 255u] + j;
    kout[out[i]] = key;
  }
  __syncthreads();
#pragma unroll
  for (int i = 0; i < kSortItems; ++i) buf[place[i]] = val[i];
  __syncthreads();
#pragma unroll
  for (int i = 0; i < kSortItems; ++i) vout[out[i]] = buf[i * kSortThreads + t];
}

// All four passes of a single tile in one launch: twelve launches would be most
// of the time of a small build.
__global__ void __launch_bounds__(kSortThreads) radix_tile_sort_kernel(uint32_t *keys, uint32_t *vals) {
  __shared__ uint32_t cnt[kSortWarps][kRadix];
  __shared__ uint32_t start[kRadix];
  __shared__ uint32_t buf[kSortTile];
  __shared__ uint32_t warp_sums[33];
  const uint32_t t = threadIdx.x, lane = t & 31u, warp = t >> 5, base = warp * (32 * kSortItems) + lane;
  uint32_t k[kSortItems], val[kSortItems], place[kSortItems];
#pragma unroll
  for (int i = 0; i < kSortItems; ++i) {
    k[i] = keys[base + 32 * i];
    val[i] = vals[base + 32 * i];
  }
  for (int shift = 0; shift < 32; shift += 8) {
    for (int i = t; i < kSortWarps * kRadix; i += kSortThreads) (&cnt[0][0])[i] = 0;
    __syncthreads();
#pragma unroll
    for (int i = 0; i < kSortItems; ++i) place[i] = rank_in_warp(cnt[warp], (k[i] >> shift) & 255u, lane);
    __syncthreads();
    uint32_t run = 0, total;
#pragma unroll
    for (int w = 0; w < kSortWarps; ++w) {
      const uint32_t x = cnt[w][t];
      cnt[w][t] = run;
      run += x;
    }
    start[t] = block_exclusive_scan(run, warp_sums, &total);
    __syncthreads();
#pragma unroll
    for (int i = 0; i < kSortItems; ++i) {
      const uint32_t d = (k[i] >> shift) & 255u;
      place[i] += start[d] + cnt[warp][d];
      buf[place[i]] = k[i];
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < kSortItems; ++i) k[i] = buf[base + 32 * i];
    __syncthreads();
#pragma unroll
    for (int i = 0; i < kSortItems; ++i) buf[place[i]] = val[i];
    __syncthreads();
#pragma unroll
    for (int i = 0; i < kSortItems; ++i) val[i] = buf[base + 32 * i];
    __syncthreads();
  }
#pragma unroll
  for (int i = 0; i < kSortItems; ++i) {
    keys[base + 32 * i] = k[i];
    vals[base + 32 * i] = val[i];
  }
}

// 4. radix tree (Karras 2012). Interior node i in [0, n-2]; leaf k is node
//    n-1+k. Common prefix length of keys i and j; equal keys compare their
//    positions; -1 outside [0, n).
__device__ __forceinline__ int delta(const uint32_t *keys, int n, int i, int j) {
  if (j < 0 || j >= n) return -1;
  const uint32_t a = keys[i], b = keys[j];
  if (a == b) return 32 + __clz((uint32_t)i ^ (uint32_t)j);
  return __clz(a ^ b);
}

__global__ void radix_tree_kernel(const uint32_t *__restrict__ keys, int n, uint32_t *left, uint32_t *right,
                                  uint32_t *parent, uint8_t *axis, uint32_t *range_lo, uint32_t *range_hi) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n - 1; i += gridDim.x * blockDim.x) {
    const int d = delta(keys, n, i, i + 1) - delta(keys, n, i, i - 1) >= 0 ? 1 : -1;
    const int dmin = delta(keys, n, i, i - d);
    // the other end of the range: exponential then binary search
    int lmax = 2;
    while (delta(keys, n, i, i + lmax * d) > dmin) lmax <<= 1;
    int l = 0;
    for (int t = lmax >> 1; t >= 1; t >>= 1)
      if (delta(keys, n, i, i + (l + t) * d) > dmin) l += t;
    const int j = i + l * d;
    const int dnode = delta(keys, n, i, j);
    // split: the last position sharing more than dnode prefix bits with i
    int s = 0;
    for (int div = 2;; div <<= 1) {
      const int t = (l + div - 1) / div;
      if (delta(keys, n, i, i + (s + t) * d) > dnode) s += t;
      if (t <= 1) break;
    }
    const int g = i + s * d + min(d, 0);
    const int lo = min(i, j), hi = max(i, j);
    const uint32_t lc = lo == g ? (uint32_t)(n - 1 + g) : (uint32_t)g;
    const uint32_t rc = hi == g + 1 ? (uint32_t)(n - 1 + g + 1) : (uint32_t)(g + 1);
    left[i] = lc;
    right[i] = rc;
    range_lo[i] = (uint32_t)lo;  // the node's leaves: sorted triangles lo..hi
    range_hi[i] = (uint32_t)hi;
    parent[lc] = (uint32_t)i;
    parent[rc] = (uint32_t)i;
    // split axis: the highest bit in which the range's end codes differ
    const uint32_t x = keys[lo] ^ keys[hi];
    uint8_t ax = 0;
    if (x) {
      const int bit = 31 - __clz(x);  // Morton bit 3m+2 = x, 3m+1 = y, 3m = z
      ax = (uint8_t)(bit % 3 == 2 ? 0 : (bit % 3 == 1 ? 1 : 2));
    }
    axis[i] = ax;
  }
}

// 5. boxes bottom-up, and the leaf choice. A subtree covers a contiguous range
//    of the sorted triangles, so it can become one leaf over that range. With
//    node and triangle test cost 1 (as the host builder), cost(x) =
//    min(area(x) * count(x) if count(x) <= leaf_max, area(x) + cost(left) +
//    cost(right)), a radix leaf costing its area; whole[x] = 1 where the leaf
//    is not dearer. Nothing above a subtree of more than leaf_max triangles
//    asks for its cost.
struct TreeArgs {
  int n;
  const uint32_t *ids, *left, *right, *parent, *rlo, *rhi;
  const Box3 *tbox;
  Box3 *box;
  uint32_t lmax;
  float *cost;
  uint8_t *whole;
  uint4 *open;
  uint32_t *arrived;
};

// Surface area in double (as the host's cost model computes it).
__device__ __forceinline__ double area_double(const Box3 &b) {
  const double ex = (double)b.hi[0] - (double)b.lo[0];
  const double ey = (double)b.hi[1] - (double)b.lo[1];
  const double ez = (double)b.hi[2] - (double)b.lo[2];
  return 2.0 * (ex * ey + ey * ez + ez * ex);
}
// The same in float: extents >= 0, so every term and sum is; relative error at
// most 5 units of 2^-24 away from overflow and underflow.
__device__ __forceinline__ float area_float(const Box3 &b) {
  const float ex = b.hi[0] - b.lo[0], ey = b.hi[1] - b.lo[1], ez = b.hi[2] - b.lo[2];
  return 2.0f * (ex * ey + ey * ez + ez * ex);
}
// cost(x) in double, x a node over at most 16 triangles, from the choices
// already made below it. A stack of its own (at most 15 interior nodes deep),
// not recursion: the call stack is small.
__device__ __noinline__ double cost_double(const TreeArgs &T, uint32_t x) {
  uint32_t id[17];
  double part[17];
  uint8_t next[17];
  int sp = 0;
  id[0] = x;
  next[0] = 0;
  double r = 0.0;
  while (sp >= 0) {
    const uint32_t y = id[sp];
    if (next[sp] == 0) {
      const double a = area_double(load_box_l2(T.box + y));
      const bool leaf = y >= (uint32_t)(T.n - 1);
      if (leaf || *(volatile uint8_t *)(T.whole + y) || sp == 16) {
        r = leaf ? a : a * (double)(T.rhi[y] - T.rlo[y] + 1u);
        --sp;
        continue;
      }
      part[sp] = a;
    } else {
      part[sp] += r;
      if (next[sp] == 2) {
        r = part[sp--];
        continue;
      }
    }
    id[sp + 1] = next[sp] == 0 ? T.left[y] : T.right[y];
    next[sp + 1] = 0;
    ++next[sp];
    ++sp;
  }
  return r;
}
// whether node p (box b) becomes one leaf of cnt triangles: the double
// comparison, taken only where float costs are too close to tell
__device__ __noinline__ bool leaf_is_cheaper(const TreeArgs &T, const Box3 &b, uint32_t cnt, uint32_t l, uint32_t r) {
  const double a = area_double(b);
  const double cl = cost_double(T, l), cr = cost_double(T, r);
  return a * (double)cnt <= a + cl + cr;
}

// Half the area, +inf where it overflows (also where an extent does and another is
// 0): whoever compares it then takes the boxes.
__device__ __forceinline__ float half_area(const Box3 &b) {
  const float ex = b.hi[0] - b.lo[0], ey = b.hi[1] - b.lo[1], ez = b.hi[2] - b.lo[2];
  const float h = ex * ey + ey * ez + ez * ex;
  return h >= 0.0f ? h : INFINITY;
}
// What a climb carries of a node and keeps of it in shared memory.
struct Made {
  Box3 b;
  float cost;
  float open;  // half area, or -1: a logical leaf
};
// Box of node p from its children's, and where the subtree is small enough the
// leaf choice (the children's costs only count for such a subtree).
__device__ __forceinline__ Made make_node(const TreeArgs &T, uint32_t p, uint32_t l, uint32_t r, uint32_t cnt,
                                          const Made &ml, const Made &mr) {
  const Box3 &b0 = ml.b, &b1 = mr.b;
  Made m;
  Box3 &b = m.b;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    b.lo[a] = fminf(b0.lo[a], b1.lo[a]);
    b.hi[a] = fmaxf(b0.hi[a], b1.hi[a]);
  }
  store_box(T.box + p, b);
  T.open[p] = make_uint4(l, r, __float_as_uint(ml.open), __float_as_uint(mr.open));
  m.cost = 0.0f;
  m.open = half_area(b);
  if (cnt > T.lmax) return m;
  const float a = area_float(b), leaf = a * (float)cnt, split = a + ml.cost + mr.cost;
  bool w = leaf <= split;
  // the terms of a subtree of at most 16 triangles carry at most 5 + 16 units
  // of 2^-24 each way: 2^-18 leaves a margin of three
  const float near = 3.8147e-06f * split;
  if (!(fabsf(leaf - split) > near) || !(split < 1e37f) || !(a > 1e-30f)) w = leaf_is_cheaper(T, b, cnt, l, r);
  T.whole[p] = w ? 1 : 0;
  m.cost = w ? leaf : split;
  T.cost[p] = m.cost;
  if (w) m.open = -1.0f;
  return m;
}

// A CTA takes kBoxTile consecutive leaves. A node whose leaves all lie in the
// tile has its number in the tile's range too (Karras: it is one end of its
// leaves' range), so those nodes, all but a few per tile, are climbed in shared
// memory; the rest climb through L2.
constexpr int kBoxTile = 256;
__global__ void __launch_bounds__(kBoxTile) boxes_kernel(TreeArgs T) {
  __shared__ Box3 leaf_box[kBoxTile];
  __shared__ Made made[kBoxTile];
  __shared__ uint32_t s_left[kBoxTile], s_right[kBoxTile], s_parent[kBoxTile], s_lo[kBoxTile], s_hi[kBoxTile];
  __shared__ uint32_t s_arrived[kBoxTile];
  const uint32_t first_leaf = (uint32_t)(T.n - 1), t = threadIdx.x;
  const uint32_t t0 = blockIdx.x * kBoxTile;
  {
    const uint32_t i = t0 + t, t1 = t0 + kBoxTile - 1;
    s_arrived[t] = 0;
    if (i < first_leaf) {
      s_left[t] = T.left[i];
      s_right[t] = T.right[i];
      s_parent[t] = T.parent[i];
      s_lo[t] = T.rlo[i];
      s_hi[t] = T.rhi[i];
    }
    uint32_t p = kNone, node = first_leaf + i;
    auto leaf_made = [](const Box3 &b) { return Made{b, area_float(b), -1.0f}; };
    Made me{};
    if (i < (uint32_t)T.n) {
      const float2 *tb = reinterpret_cast<const float2 *>(T.tbox + T.ids[i]);
      me = leaf_made(unpack_box(__ldg(tb), __ldg(tb + 1), __ldg(tb + 2)));
      leaf_box[t] = me.b;
      store_box(T.box + node, me.b);
      p = T.parent[node];
    }
    __syncthreads();
    // at most one thread continues past each node: the second to arrive. It
    // carries its own node and fetches its sibling.
    while (p != kNone && p - t0 < (uint32_t)kBoxTile && s_lo[p - t0] >= t0 && s_hi[p - t0] <= t1) {
      const uint32_t j = p - t0;
      __threadfence_block();
      if (atomicAdd(s_arrived + j, 1u) == 0u) {
        p = kNone;
        break;
      }
      __threadfence_block();
      const uint32_t l = s_left[j], r = s_right[j], cnt = s_hi[j] - s_lo[j] + 1u;
      const bool left = l == node;
      const uint32_t sib = left ? r : l;
      const Made other = sib >= first_leaf ? leaf_made(leaf_box[sib - first_leaf - t0]) : made[sib - t0];
      me = make_node(T, p, l, r, cnt, left ? me : other, left ? other : me);
      made[j] = me;
      node = p;
      p = s_parent[j];
    }
    while (p != kNone) {
      // none of these depend on the arrival: in flight together with it
      const uint32_t l = __ldg(T.left + p), r = __ldg(T.right + p), lo = __ldg(T.rlo + p), hi = __ldg(T.rhi + p);
      const uint32_t up = __ldg(T.parent + p);
      __threadfence();
      if (atomicAdd(T.arrived + p, 1u) == 0u) break;
      __threadfence();
      const bool left = l == node;
      const uint32_t sib = left ? r : l, cnt = hi - lo + 1u;
      Made other;
      other.b = load_box_l2(T.box + sib);
      if (sib >= first_leaf) {
        other = leaf_made(other.b);
      } else {
        const bool w = __ldcg(T.whole + sib) != 0;
        other.cost = cnt <= T.lmax ? __ldcg(T.cost + sib) : 0.0f;
        other.open = w ? -1.0f : half_area(other.b);
      }
      me = make_node(T, p, l, r, cnt, left ? me : other, left ? other : me);
      node = p;
      p = up;
    }
  }
}

scion_status fail(cudaError_t e, std::string *err) {
  *err = cudaGetErrorString(e);
  return e == cudaErrorMemoryAllocation ? SCION_ERR_OOM : SCION_ERR_CUDA;
}

int grid_for(uint64_t n, int threads) {
  return (int)std::max<uint64_t>(1, std::min<uint64_t>((n + threads - 1) / threads, 152ull * 16));
}

}  // namespace

namespace {

// The library's scratch pool of the current device, created on first use; null
// where the device has no memory pools or it cannot be created.
cudaMemPool_t scratch_pool() {
  constexpr int kMaxDevices = 64;
  static std::mutex mu;
  static cudaMemPool_t pools[kMaxDevices] = {};
  static bool tried[kMaxDevices] = {};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return nullptr;
  std::lock_guard<std::mutex> lk(mu);
  if (!tried[dev]) {
    tried[dev] = true;
    int supported = 0;
    cudaDeviceGetAttribute(&supported, cudaDevAttrMemoryPoolsSupported, dev);
    cudaMemPoolProps props{};
    props.allocType = cudaMemAllocationTypePinned;
    props.location.type = cudaMemLocationTypeDevice;
    props.location.id = dev;
    cudaMemPool_t p = nullptr;
    if (supported && cudaMemPoolCreate(&p, &props) == cudaSuccess) {
      uint64_t kept = kScratchKept;
      if (cudaMemPoolSetAttribute(p, cudaMemPoolAttrReleaseThreshold, &kept) == cudaSuccess) pools[dev] = p;
      else cudaMemPoolDestroy(p);
    }
    cudaGetLastError();
  }
  return pools[dev];
}

}  // namespace

void release_scratch() {
  if (const cudaMemPool_t pool = scratch_pool()) cudaMemPoolTrimTo(pool, 0);
}

cudaError_t device_malloc(void **p, size_t bytes) {
  cudaError_t e = cudaMalloc(p, bytes);
  if (e == cudaErrorMemoryAllocation) {
    cudaGetLastError();
    release_scratch();
    e = cudaMalloc(p, bytes);
  }
  return e;
}

Arena::~Arena() {
  if (!base_) return;
  if (pooled_) cudaFreeAsync(base_, stream_);
  else cudaFree(base_);
}

cudaError_t Arena::commit() {
  void *q = nullptr;
  const cudaError_t e = device_malloc(&q, used_ ? used_ : 256);
  base_ = static_cast<char *>(e == cudaSuccess ? q : nullptr);
  used_ = 0;
  return e;
}

cudaError_t Arena::commit(cudaStream_t stream) {
  const cudaMemPool_t pool = scratch_pool();
  if (!pool) return commit();
  void *q = nullptr;
  const cudaError_t e = cudaMallocFromPoolAsync(&q, used_ ? used_ : 256, pool, stream);
  if (e != cudaSuccess) {  // e.g. the device is full but for what the pool keeps
    cudaGetLastError();
    release_scratch();
    return commit();
  }
  base_ = static_cast<char *>(q);
  used_ = 0;
  pooled_ = true;
  stream_ = stream;
  return cudaSuccess;
}

scion_status lbvh_build_tree(const float *d_verts, uint64_t n_verts, const uint32_t *d_indices, uint64_t n_tris,
                             uint32_t leaf_max, cudaStream_t s, LbvhTree *out, std::string *err) {
  out->nv = 0;
  out->gpu_ms = 0.0;
  if (n_tris == 0) return SCION_OK;
  const uint32_t n = (uint32_t)n_tris;
  const uint32_t tiles = (n + kSortTile - 1) / kSortTile;
  const size_t npad = (size_t)tiles * kSortTile, nn_max = 2 * (size_t)n - 1;
  Box3 *tbox, *box;
  uint32_t *keys[2], *vals[2], *hist, *totals, *cb, *nvalid, *left, *right, *parent, *arrived, *rlo, *rhi;
  uint8_t *axis, *whole;
  float *cost;
  uint4 *open;
  cudaError_t e;
#define SCION_LB(call)              \
  do {                              \
    e = (call);                     \
    if (e != cudaSuccess) return fail(e, err); \
  } while (0)
  // tree and scratch, sized for n valid triangles: one allocation, the result's
  Arena &mem = out->memory;
  for (int pass = 0; pass < 2; ++pass) {  // sizes, then addresses
    if (pass) SCION_LB(mem.commit(s));
    mem.take(&cb, 8);  // centroid bounds, valid count, bad index flag
    mem.take(&tbox, n);
    for (int b = 0; b < 2; ++b) {
      mem.take(&keys[b], npad);
      mem.take(&vals[b], npad);
    }
    mem.take(&hist, (size_t)kRadix * tiles);
    mem.take(&totals, kRadix);
    mem.take(&left, n);
    mem.take(&right, n);
    mem.take(&rlo, n);
    mem.take(&rhi, n);
    mem.take(&axis, n);
    mem.take(&whole, n);
    mem.take(&box, nn_max);
    mem.take(&parent, nn_max);
    mem.take(&arrived, n);
    mem.take(&cost, n);
    mem.take(&open, n);
  }
  nvalid = cb + 6;
  int *bad_index = reinterpret_cast<int *>(cb + 7);
  cudaEvent_t ev0, ev1;
  SCION_LB(cudaEventCreate(&ev0));
  SCION_LB(cudaEventCreate(&ev1));
  struct EvGuard {
    cudaEvent_t a, b;
    ~EvGuard() {
      cudaEventDestroy(a);
      cudaEventDestroy(b);
    }
  } evg{ev0, ev1};
  SCION_LB(cudaEventRecord(ev0, s));
  SCION_LB(cudaMemsetAsync(cb, 0xFF, 3 * sizeof(uint32_t), s));
  SCION_LB(cudaMemsetAsync(cb + 3, 0, 5 * sizeof(uint32_t), s));
  launch_index_check(d_indices, n_tris, n_verts, bad_index, s);
  SCION_LB(cudaGetLastError());
  // padding keys sort after every real key (and after the invalid ones)
  SCION_LB(cudaMemsetAsync(keys[0], 0xFF, npad * sizeof(uint32_t), s));
  SCION_LB(cudaMemsetAsync(vals[0], 0xFF, npad * sizeof(uint32_t), s));
  tri_bounds_kernel<<<std::min(grid_for(n, kBoundsThreads), 152 * 6), kBoundsThreads, 0, s>>>(d_verts, d_indices, n,
                                                                                             tbox, cb, nvalid, bad_index);
  SCION_LB(cudaGetLastError());
  morton_kernel<<<grid_for(n, 256), 256, 0, s>>>(d_verts, d_indices, tbox, n, cb, keys[0], vals[0],
                                               bad_index);
  SCION_LB(cudaGetLastError());
  int cur = 0;
  if (tiles == 1) {
    radix_tile_sort_kernel<<<1, kSortThreads, 0, s>>>(keys[0], vals[0]);
    SCION_LB(cudaGetLastError());
  }
  for (int shift = 0; shift < 32 && tiles > 1; shift += 8) {
    radix_hist_kernel<<<tiles, kSortThreads, 0, s>>>(keys[cur], shift, hist, tiles);
    radix_scan_kernel<<<kRadix, kSortThreads, 0, s>>>(hist, tiles, totals);
    radix_scatter_kernel<<<tiles, kSortThreads, 0, s>>>(keys[cur], vals[cur], keys[cur ^ 1], vals[cur ^ 1], shift,
                                                         hist, totals, tiles);
    SCION_LB(cudaGetLastError());
    cur ^= 1;
  }
  uint32_t found[2] = {0, 0};  // valid triangles, bad index flag
  SCION_LB(cudaMemcpyAsync(found, nvalid, sizeof(found), cudaMemcpyDeviceToHost, s));
  SCION_LB(cudaStreamSynchronize(s));
  if (found[1]) {
    *err = "scion_build_gpu: a vertex index is out of range";
    return SCION_ERR_INVALID_ARG;
  }
  const uint32_t nv = found[0];
  out->ids = vals[cur];
  if (nv == 0) {
    SCION_LB(cudaEventRecord(ev1, s));
    SCION_LB(cudaEventSynchronize(ev1));
    return SCION_OK;
  }
  const size_t nn = 2 * (size_t)nv - 1;
  SCION_LB(cudaMemsetAsync(parent, 0xFF, nn * sizeof(uint32_t), s));
  SCION_LB(cudaMemsetAsync(arrived, 0, nv * sizeof(uint32_t), s));
  SCION_LB(cudaMemsetAsync(whole, 0, nv, s));
  if (nv > 1) {
    radix_tree_kernel<<<grid_for(nv - 1, 256), 256, 0, s>>>(keys[cur], (int)nv, left, right, parent, axis, rlo,
                                                             rhi);
    SCION_LB(cudaGetLastError());
  }
  const TreeArgs T{(int)nv, vals[cur], left, right, parent, rlo, rhi, tbox, box, leaf_max ? leaf_max : 1u,
                   cost,    whole,     open, arrived};
  // a CTA per tile: one that climbs through L2 must not hold up another tile
  boxes_kernel<<<(nv + kBoxTile - 1) / kBoxTile, kBoxTile, 0, s>>>(T);
  SCION_LB(cudaGetLastError());
  SCION_LB(cudaEventRecord(ev1, s));
  SCION_LB(cudaStreamSynchronize(s));
  float ms = 0.f;
  SCION_LB(cudaEventElapsedTime(&ms, ev0, ev1));
  out->gpu_ms = ms;
#undef SCION_LB
  out->nv = nv;
  out->left = left;
  out->right = right;
  out->rlo = rlo;
  out->rhi = rhi;
  out->axis = axis;
  out->whole = whole;
  out->box = box;
  out->open = open;
  return SCION_OK;
}

scion_status lbvh_download(const LbvhTree &t, cudaStream_t s, LogicalBVH *out, std::string *err) {
  out->nodes.clear();
  out->prims.clear();
  const uint32_t nv = t.nv;
  if (nv == 0) return SCION_OK;
  const size_t nn = 2 * (size_t)nv - 1;
  std::vector<uint32_t> hl(nv), hr(nv), ids(nv), hrl(nv), hrh(nv);
  std::vector<uint8_t> hax(nv), whole(nv);
  std::vector<Box3> hbox(nn);
  cudaError_t e = cudaSuccess;
#define SCION_DL(dst, src, bytes) \
  if (e == cudaSuccess) e = cudaMemcpyAsync(dst, src, bytes, cudaMemcpyDeviceToHost, s)
  SCION_DL(ids.data(), t.ids, nv * sizeof(uint32_t));
  SCION_DL(hl.data(), t.left, nv * sizeof(uint32_t));
  SCION_DL(hr.data(), t.right, nv * sizeof(uint32_t));
  SCION_DL(hax.data(), t.axis, nv);
  SCION_DL(whole.data(), t.whole, nv);
  SCION_DL(hrl.data(), t.rlo, nv * sizeof(uint32_t));
  SCION_DL(hrh.data(), t.rhi, nv * sizeof(uint32_t));
  SCION_DL(hbox.data(), t.box, nn * sizeof(Box3));
#undef SCION_DL
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  if (e != cudaSuccess) return fail(e, err);
  // Logical tree, depth first from the root.
  out->prims = std::move(ids);
  out->nodes.reserve(nn);
  struct Item {
    uint32_t src, dst;  // node of the radix tree, node of the logical tree
  };
  std::vector<Item> todo;
  auto emit = [&](uint32_t src) {
    LNode d{};
    d.box = hbox[src];
    const uint32_t id = (uint32_t)out->nodes.size();
    if (src + 1 >= nv) {  // a leaf of the radix tree: one triangle
      d.first = src - (nv - 1);
      d.count = 1;
    } else if (whole[src]) {
      d.first = hrl[src];
      d.count = hrh[src] - hrl[src] + 1;
    } else {
      d.axis = hax[src];
      todo.push_back(Item{src, id});
    }
    out->nodes.push_back(d);
    return id;
  };
  emit(0);
  while (!todo.empty()) {
    const Item it = todo.back();
    todo.pop_back();
    const uint32_t l = emit(hl[it.src]);
    const uint32_t r = emit(hr[it.src]);
    out->nodes[it.dst].left = l;
    out->nodes[it.dst].right = r;
  }
  return SCION_OK;
}

scion_status lbvh_build(const float *d_verts, uint64_t n_verts, const uint32_t *d_indices, uint64_t n_tris,
                        uint32_t leaf_max, cudaStream_t s, LogicalBVH *out, double *gpu_ms, std::string *err) {
  out->nodes.clear();
  out->prims.clear();
  *gpu_ms = 0.0;
  LbvhTree t;
  scion_status st = lbvh_build_tree(d_verts, n_verts, d_indices, n_tris, leaf_max, s, &t, err);
  if (st != SCION_OK) return st;
  *gpu_ms = t.gpu_ms;
  return lbvh_download(t, s, out, err);
}

}  // namespace scion
