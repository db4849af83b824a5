// GPU construction of the logical BVH2 (the "construction" phase that the
// paper keeps apart from the layout build, Section 5 footnote and Section 5.1
// two-phase construction; Section 2: topology is orthogonal to layout).
//
// Linear BVH: triangles are ordered along a 30-bit Morton curve of their box
// centres (Lauterbach et al. 2009), the binary radix tree over the sorted
// codes is built with one thread per interior node (Karras 2012), and boxes
// are computed bottom-up. A subtree of at most leaf_max triangles (a
// contiguous range of the sorted order) becomes one leaf where the surface
// area heuristic prefers it to the subtree's best split. The result is the
// same LogicalBVH the host SAH builder produces, so every packer and layout
// applies unchanged.
#pragma once

#include <cuda_runtime.h>

#include <string>
#include <vector>

#include "builder.h"

namespace scion {

// One device allocation cut into arrays: take every array (which only adds up
// sizes), commit, take them again in the same order (which gives addresses).
// cudaMalloc and cudaFree of a few MB cost 35 us each here, of hundreds of MB
// 50 and 200 us: more than most kernels of a build. commit(stream) allocates
// scratch for the duration of a call on that stream, from a memory pool of the
// library's own that keeps up to kScratchKept bytes per device between calls
// (the driver gives the rest back, and hands the pool's memory to any thread
// or stream in order); commit() allocates a result with cudaMalloc. Freed with
// the object unless released. Every array starts at a multiple of 256 bytes: the
// kernels' 32-byte node loads rely on it.
constexpr uint64_t kScratchKept = 512ull << 20;
class Arena {
 public:
  Arena() = default;
  Arena(const Arena &) = delete;
  Arena &operator=(const Arena &) = delete;
  ~Arena();
  template <typename T>
  void take(T **p, uint64_t count) {
    if (base_) *p = reinterpret_cast<T *>(base_ + used_);
    used_ += (count * sizeof(T) + 255) & ~255ull;
  }
  cudaError_t commit();
  cudaError_t commit(cudaStream_t stream);
  void *release() {  // of a commit() without a stream
    void *q = base_;
    base_ = nullptr;
    return q;
  }

 private:
  char *base_ = nullptr;
  uint64_t used_ = 0;
  bool pooled_ = false;
  cudaStream_t stream_ = nullptr;
};

// Gives back what the current device's pool keeps and no call uses.
void release_scratch();
// cudaMalloc, once more without what the pool keeps where the device is full.
cudaError_t device_malloc(void **p, size_t bytes);

// The logical BVH2 as the GPU builds it, left in device memory: the binary
// radix tree over the nv valid triangles in Morton order. Interior node i in
// [0, nv-2] has children left[i], right[i]; node ids >= nv-1 are radix
// leaves (leaf k = node nv-1+k holds the sorted triangle ids[k]). An
// interior node with whole[i] = 1 is a logical leaf over the sorted
// triangles rlo[i]..rhi[i]; the logical tree is what is reachable from node
// 0 without entering such a node. open[i] of an interior node that is not a
// leaf: its children and their half areas, -1 for a logical leaf: what opening
// the node takes, in one load. Boxes: one per node (2nv-1 nodes), 8-byte
// aligned. Node 0 is the root (a radix leaf when nv = 1). Owns its device
// memory; freed with the object.
struct LbvhTree {
  uint32_t nv = 0;
  const uint32_t *ids = nullptr;
  const uint32_t *left = nullptr, *right = nullptr, *rlo = nullptr, *rhi = nullptr;
  const uint8_t *axis = nullptr, *whole = nullptr;
  const Box3 *box = nullptr;
  const uint4 *open = nullptr;
  double gpu_ms = 0.0;  // device time of the build kernels
  Arena memory;
};

// Build from device vertex (float[n_verts][3]) and optional device index
// (u32[n_tris][3]) arrays. Triangles with a non-finite vertex are left out. An
// index out of range gives INVALID_ARG, found on the GPU before any kernel
// reads through the indices.
// Synchronises `stream` before returning.
scion_status lbvh_build_tree(const float *d_verts, uint64_t n_verts, const uint32_t *d_indices, uint64_t n_tris,
                             uint32_t leaf_max, cudaStream_t stream, LbvhTree *out, std::string *err);

// The tree in host memory, as the host packers take it.
scion_status lbvh_download(const LbvhTree &t, cudaStream_t stream, LogicalBVH *out, std::string *err);

// Both steps. *gpu_ms receives the device time of the build kernels (bounds,
// codes, sort, tree, boxes, leaf choice), without the download.
scion_status lbvh_build(const float *d_verts, uint64_t n_verts, const uint32_t *d_indices, uint64_t n_tris,
                        uint32_t leaf_max, cudaStream_t stream, LogicalBVH *out, double *gpu_ms, std::string *err);

}  // namespace scion
