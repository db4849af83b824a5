// Backward pass of the closest-hit query: with the traversal's discrete choice
// (which triangle each ray hit) held fixed, carry dL/d(t, u, v) of every hit
// ray to the hit triangle's three vertices and to the ray's origin and
// direction. The paper has no gradient; this follows from differentiating the
// hit-point identity o + t d = (1-u-v) p0 + u p1 + v p2 (the barycentric
// convention b1 = u, b2 = v of the closest-hit listing in App. G).
//
// With J = [d | -(p1-p0) | -(p2-p0)] and g = (dL/dt, dL/du, dL/dv), lambda
// solves J^T lambda = g; then dL/do = -lambda, dL/dd = -t lambda,
// dL/dp0 = (1-u-v) lambda, dL/dp1 = u lambda, dL/dp2 = v lambda.
//
// One thread per ray (grid-stride). The 3x3 solve runs in single precision
// (Cramer's rule) followed by one step of iterative refinement whose residual
// g - J^T lambda is formed to twice single precision: the columns of J as
// exact pairs of floats (TwoDiff, Knuth), products as exact pairs (one fma
// each), summed with the rounding errors carried along (the compensated dot
// product of Ogita, Rump and Oishi, 2005). The error after the step is of the
// order of the square of the first solve's, so lambda comes out accurate to
// the last bit or so of a float for any system that is not extremely ill
// conditioned. FP64 has a small fraction of the FP32 rate here: with the
// residual in doubles (about 45 FP64 operations a hit) that pipe was 81 % busy.
// A singular or
// non-finite single-precision solve, and gradients so small or large that the
// pairs could underflow or overflow, take the double-precision solve.
//
// The nine vertex contributions are added with FP32 atomics, a vertex's three
// as a pair and a single (row i of the float[n][3] array starts at 12 i bytes:
// the 8-byte aligned pair is its first two elements when i is even, its last
// two when it is odd).
#include <cuda_runtime.h>
#include <stdint.h>

#include "../../include/scion.h"
#include "backward.h"

namespace scion {

namespace {

__device__ __forceinline__ void cross3(const double *a, const double *b, double *c) {
  c[0] = a[1] * b[2] - a[2] * b[1];
  c[1] = a[2] * b[0] - a[0] * b[2];
  c[2] = a[0] * b[1] - a[1] * b[0];
}

__device__ __forceinline__ double dot3(const double *a, const double *b) {
  return a[0] * b[0] + a[1] * b[1] + a[2] * b[2];
}

__device__ __forceinline__ void cross3f(const float *a, const float *b, float *c) {
  c[0] = fmaf(a[1], b[2], -a[2] * b[1]);
  c[1] = fmaf(a[2], b[0], -a[0] * b[2]);
  c[2] = fmaf(a[0], b[1], -a[1] * b[0]);
}

struct Pair {  // an unevaluated sum hi + lo
  float hi, lo;
};

// x - y exactly (TwoDiff; no overflow)
__device__ __forceinline__ Pair two_diff(float x, float y) {
  const float d = __fsub_rn(x, y);
  const float t = __fsub_rn(d, x);
  return {d, __fsub_rn(__fsub_rn(x, __fsub_rn(d, t)), __fadd_rn(y, t))};
}

// acc -= a * m, the rounding errors of the product and of the sum going to err
__device__ __forceinline__ void sub_product(float a, float m, float &acc, float &err) {
  const float p = __fmul_rn(a, m), e = fmaf(a, m, -p);
  const float s = __fsub_rn(acc, p);
  const float t = __fsub_rn(s, acc);
  err = __fadd_rn(err, __fsub_rn(__fsub_rn(__fsub_rn(acc, __fsub_rn(s, t)), __fadd_rn(p, t)), e));
  acc = s;
}

// g - c . l to about twice single precision, c given in pairs
__device__ __forceinline__ float residual(const Pair *c, const float *l, float g) {
  float acc = g, err = 0.0f;
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    sub_product(c[k].hi, l[k], acc, err);
    err = fmaf(-c[k].lo, l[k], err);
  }
  return __fadd_rn(acc, err);
}

// lambda with J^T lambda = (gt, gu, gv), J = [c0 | c1 | c2]: single-precision
// Cramer's rule, then one refinement step lambda += J^-T (g - J^T lambda).
// False when the single-precision system is singular, the result is not
// finite or the gradients leave the range of the pairs.
__device__ __forceinline__ bool solve_refined(const Pair *c0, const Pair *c1, const Pair *c2, float gt, float gu,
                                              float gv, float *lam) {
  const float gmax = fmaxf(fmaxf(fabsf(gt), fabsf(gu)), fabsf(gv));
  if (!(gmax == 0.0f || (gmax > 1e-28f && gmax < 1e28f))) return false;
  const float f0[3] = {c0[0].hi, c0[1].hi, c0[2].hi};
  const float f1[3] = {c1[0].hi, c1[1].hi, c1[2].hi};
  const float f2[3] = {c2[0].hi, c2[1].hi, c2[2].hi};
  float x12[3], x20[3], x01[3];
  cross3f(f1, f2, x12);
  cross3f(f2, f0, x20);
  cross3f(f0, f1, x01);
  const float det = fmaf(f0[0], x12[0], fmaf(f0[1], x12[1], f0[2] * x12[2]));
  if (!(det != 0.0f) || !isfinite(det)) return false;
  const float inv = 1.0f / det;
  float l0[3];
  for (int k = 0; k < 3; ++k) l0[k] = fmaf(gt, x12[k], fmaf(gu, x20[k], gv * x01[k])) * inv;
  const float s0 = residual(c0, l0, gt), s1 = residual(c1, l0, gu), s2 = residual(c2, l0, gv);
  for (int k = 0; k < 3; ++k) {
    lam[k] = l0[k] + fmaf(s0, x12[k], fmaf(s1, x20[k], s2 * x01[k])) * inv;
    if (!isfinite(lam[k])) return false;
  }
  return true;
}

// grad_verts[vid] += w * l. PAIRED: the array starts on an 8-byte boundary.
template <bool PAIRED>
__device__ __forceinline__ void add_vertex(float *grad_verts, uint32_t vid, float w, const float *l) {
  float *g = grad_verts + 3 * (size_t)vid;
  const float x = w * l[0], y = w * l[1], z = w * l[2];
  if (!PAIRED) {
    atomicAdd(g, x);
    atomicAdd(g + 1, y);
    atomicAdd(g + 2, z);
    return;
  }
  const bool odd = (vid & 1u) != 0u;
  atomicAdd(reinterpret_cast<float2 *>(g + (odd ? 1 : 0)), odd ? make_float2(y, z) : make_float2(x, y));
  atomicAdd(g + (odd ? 0 : 2), odd ? x : z);
}

// PACKED: the three gradients of a ray lie together (strides of 3 from grad[0]).
template <bool PAIRED, bool PACKED>
__global__ void __launch_bounds__(256) backward_kernel(BackwardArgs a) {
  const unsigned long long stride = (unsigned long long)gridDim.x * blockDim.x;
  const uint32_t lane = threadIdx.x & 31u;
  for (unsigned long long b = (unsigned long long)blockIdx.x * blockDim.x + (threadIdx.x & ~31u); b < a.n; b += stride) {
    const unsigned long long i = b + lane;
    uint4 h = make_uint4(0, 0, 0, 0xFFFFFFFFu);
    if (i < a.n) h = __ldg(reinterpret_cast<const uint4 *>(a.hits) + i);
    const uint32_t prim = h.w;
    bool valid = prim < a.n_tris;
    float lf[3] = {0.f, 0.f, 0.f};
    uint32_t vid[3] = {0, 0, 0};
    if (valid) {
      if (a.tri_idx) {
        vid[0] = __ldg(a.tri_idx + 3 * (size_t)prim);
        vid[1] = __ldg(a.tri_idx + 3 * (size_t)prim + 1);
        vid[2] = __ldg(a.tri_idx + 3 * (size_t)prim + 2);
      } else {
        vid[0] = 3 * prim;
        vid[1] = 3 * prim + 1;
        vid[2] = 3 * prim + 2;
      }
      const float4 p0 = __ldg(a.verts + vid[0]), p1 = __ldg(a.verts + vid[1]), p2 = __ldg(a.verts + vid[2]);
      const float4 rd = __ldg(reinterpret_cast<const float4 *>(a.rays) + 2 * i + 1);
      // columns of J, each an exact pair
      const Pair c0[3] = {{rd.x, 0.f}, {rd.y, 0.f}, {rd.z, 0.f}};
      const Pair c1[3] = {two_diff(p0.x, p1.x), two_diff(p0.y, p1.y), two_diff(p0.z, p1.z)};
      const Pair c2[3] = {two_diff(p0.x, p2.x), two_diff(p0.y, p2.y), two_diff(p0.z, p2.z)};
      float g[3];
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        if (PACKED) g[k] = __ldg(a.grad[0] + 3 * i + k);
        else g[k] = a.grad[k] ? __ldg(a.grad[k] + (long long)i * a.stride[k]) : 0.0f;
      }
      const float gt = g[0], gu = g[1], gv = g[2];
      if (!solve_refined(c0, c1, c2, gt, gu, gv, lf)) {
        // the columns in double: differences of two floats
        const double e0[3] = {rd.x, rd.y, rd.z};
        const double e1[3] = {(double)p0.x - p1.x, (double)p0.y - p1.y, (double)p0.z - p1.z};
        const double e2[3] = {(double)p0.x - p2.x, (double)p0.y - p2.y, (double)p0.z - p2.z};
        double x12[3], x20[3], x01[3];
        cross3(e1, e2, x12);
        cross3(e2, e0, x20);
        cross3(e0, e1, x01);
        const double det = dot3(e0, x12);
        if (det == 0.0) valid = false;
        for (int k = 0; k < 3; ++k)
          lf[k] = valid ? (float)(((double)gt * x12[k] + (double)gu * x20[k] + (double)gv * x01[k]) / det) : 0.f;
      }
    }
    const float t = valid ? __uint_as_float(h.x) : 0.f, u = __uint_as_float(h.y), v = __uint_as_float(h.z);
    if (a.grad_rays && i < a.n) {
      float4 *gr = reinterpret_cast<float4 *>(a.grad_rays) + 2 * i;
      gr[0] = valid ? make_float4(-lf[0], -lf[1], -lf[2], 0.f) : make_float4(0.f, 0.f, 0.f, 0.f);
      gr[1] = valid ? make_float4(-t * lf[0], -t * lf[1], -t * lf[2], 0.f) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
    float c[9];
    const float w[3] = {(1.0f - u) - v, u, v};
    for (int j = 0; j < 3; ++j)
      for (int k = 0; k < 3; ++k) c[3 * j + k] = valid ? w[j] * lf[k] : 0.f;
    // neighbouring rays often hit one triangle: the first lane of such a run
    // adds the run's sum (segmented sums over the warp, skipped where no lane
    // follows its neighbour)
    const uint32_t key = valid ? prim : 0xFFFFFFFFu;
    const uint32_t prev = __shfl_up_sync(0xFFFFFFFFu, key, 1);
    const bool same = valid && lane > 0 && prev == key;
    const uint32_t heads = __ballot_sync(0xFFFFFFFFu, !same);
    if (heads != 0xFFFFFFFFu) {
      const uint32_t later = heads & (0xFFFFFFFEu << lane);  // first lanes of the runs after this lane's
      const uint32_t end = later ? __ffs(later) - 1 : 32;
      for (int o = 1; o < 32; o <<= 1) {
        const bool in = lane + o < end;
#pragma unroll
        for (int k = 0; k < 9; ++k) {
          const float x = __shfl_down_sync(0xFFFFFFFFu, c[k], o);
          if (in) c[k] += x;
        }
      }
    }
    if (valid && !same) {
      for (int j = 0; j < 3; ++j) add_vertex<PAIRED>(a.grad_verts, vid[j], 1.0f, c + 3 * j);
    }
  }
}

__global__ void __launch_bounds__(256) split_hits_kernel(const uint4 *__restrict__ hits, unsigned long long n, float *t,
                                                         float *u, float *v, uint32_t *prim) {
  const unsigned long long stride = (unsigned long long)gridDim.x * blockDim.x;
  for (unsigned long long i = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
    const uint4 h = __ldg(hits + i);
    t[i] = __uint_as_float(h.x);
    u[i] = __uint_as_float(h.y);
    v[i] = __uint_as_float(h.z);
    prim[i] = h.w;
  }
}

}  // namespace

cudaError_t launch_split_hits(const uint32_t *hits, unsigned long long n, float *t, float *u, float *v, uint32_t *prim,
                              int sms, cudaStream_t s) {
  if (n == 0) return cudaSuccess;
  const unsigned long long blocks = (n + 255) / 256, most = (unsigned long long)sms * 16;
  split_hits_kernel<<<(unsigned)(blocks < most ? blocks : most), 256, 0, s>>>(reinterpret_cast<const uint4 *>(hits), n, t, u,
                                                                             v, prim);
  return cudaGetLastError();
}

cudaError_t launch_backward(const BackwardArgs &a, int sms, cudaStream_t s) {
  if (a.n == 0) return cudaSuccess;
  const unsigned long long blocks = (a.n + 255) / 256;
  const unsigned grid = (unsigned)(blocks < (unsigned long long)sms * 8 ? blocks : (unsigned long long)sms * 8);
  const bool paired = (reinterpret_cast<uintptr_t>(a.grad_verts) & 7u) == 0;
  const bool packed = a.grad[0] && a.grad[1] == a.grad[0] + 1 && a.grad[2] == a.grad[0] + 2 && a.stride[0] == 3 &&
                      a.stride[1] == 3 && a.stride[2] == 3;
  if (paired && packed) backward_kernel<true, true><<<grid, 256, 0, s>>>(a);
  else if (paired) backward_kernel<true, false><<<grid, 256, 0, s>>>(a);
  else if (packed) backward_kernel<false, true><<<grid, 256, 0, s>>>(a);
  else backward_kernel<false, false><<<grid, 256, 0, s>>>(a);
  return cudaGetLastError();
}

}  // namespace scion
