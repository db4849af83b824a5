// Closest point query on the same layouts (App. G "Closest Point Query").
//
// For a point p and a squared search radius r2, the result is the
// lexicographic minimum of (d2, id) over triangles with d2 <= r2, where d2 is
// the squared distance from p to the closest point on the triangle computed
// by the Voronoi-region method of Ericson, Real-Time Collision Detection
// (2005), Section 5.1.5, in float with a fixed order of roundings:
//   dot(x, y) = (x0*y0 + x1*y1) + x2*y2; ab = b - a, ac = c - a, ap = p - a;
//   d1 = dot(ab, ap), d2 = dot(ac, ap) -> vertex a if d1 <= 0 && d2 <= 0;
//   bp = p - b, d3 = dot(ab, bp), d4 = dot(ac, bp) -> vertex b if d3 >= 0 && d4 <= d3;
//   vc = d1*d4 - d3*d2 -> edge ab if vc <= 0 && d1 >= 0 && d3 <= 0, s = d1/(d1-d3);
//   cp = p - c, d5 = dot(ab, cp), d6 = dot(ac, cp) -> vertex c if d6 >= 0 && d5 <= d6;
//   vb = d5*d2 - d1*d6 -> edge ac if vb <= 0 && d2 >= 0 && d6 <= 0, s = d2/(d2-d6);
//   va = d3*d6 - d5*d4 -> edge bc if va <= 0 && d4-d3 >= 0 && d5-d6 >= 0,
//     s = (d4-d3)/((d4-d3)+(d5-d6)), q = b + s*(c-b);
//   else face: r = 1/((va+vb)+vc), v = vb*r, w = vc*r, clamped to >= 0 and
//     divided by v+w when that exceeds 1, q = (a + ab*v) + ac*w;
//   d2 = dot(p-q, p-q).
// The clamp keeps q inside the triangle when rounding makes the region tests
// disagree, so q lies inside every (padded, outward-rounded) box on the path
// to the triangle. The box bound is therefore safe: per axis the gap to the
// box and its square are rounded toward -inf and summed toward -inf; a box is
// entered iff that bound <= limit (1 + 2^-18) + 1e-42, limit = min(best d2,
// r2). The widening covers the rounding of the subtraction p - q and of the dot
// product (at most 5 units of 2^-24 relative, a few denormal units absolute),
// on the side of the limit, once per node or pop. The paper's "distmax" bound update is not
// used: it does not bound the distance to the nearest triangle for boxes
// that are not tight.
#pragma once

#include "trace.cuh"

namespace scion {

// Best point so far. A query starts with d2 = r2 and id = SCION_PRIM_MISS, so
// a triangle at d2 = r2 is accepted (its id is below) and one beyond is not.
struct CpBest {
  float d2, u, v;
  uint32_t id;
};

struct CpLane {
  float px, py, pz;
  CpBest b;
  uint32_t cur;
  uint32_t count, field;  // own-box layouts: the current node's primitive count and reference
  uint32_t steps;
  uint32_t err;
  unsigned long long rid;
};

__device__ __forceinline__ float cp_dot(float x0, float x1, float x2, float y0, float y1, float y2) {
  return __fadd_rn(__fadd_rn(__fmul_rn(x0, y0), __fmul_rn(x1, y1)), __fmul_rn(x2, y2));
}

// squared distance to the pinned closest point on triangle (a, b, c); (u, v)
// are the weights of b and c. The regions stay nested branches: computing all
// seven regions' operands in one sequence with selects and a single division
// measured 15 % slower (the early regions skip most of the work)
__device__ __forceinline__ float cp_triangle(float px, float py, float pz, float4 A, float4 B, float4 C,
                                             float &u, float &v) {
  const float abx = __fsub_rn(B.x, A.x), aby = __fsub_rn(B.y, A.y), abz = __fsub_rn(B.z, A.z);
  const float acx = __fsub_rn(C.x, A.x), acy = __fsub_rn(C.y, A.y), acz = __fsub_rn(C.z, A.z);
  const float apx = __fsub_rn(px, A.x), apy = __fsub_rn(py, A.y), apz = __fsub_rn(pz, A.z);
  float qx, qy, qz;
  const float d1 = cp_dot(abx, aby, abz, apx, apy, apz), d2 = cp_dot(acx, acy, acz, apx, apy, apz);
  if (d1 <= 0.0f && d2 <= 0.0f) {
    u = 0.0f; v = 0.0f;
    qx = A.x; qy = A.y; qz = A.z;
  } else {
    const float bpx = __fsub_rn(px, B.x), bpy = __fsub_rn(py, B.y), bpz = __fsub_rn(pz, B.z);
    const float d3 = cp_dot(abx, aby, abz, bpx, bpy, bpz), d4 = cp_dot(acx, acy, acz, bpx, bpy, bpz);
    const float vc = __fsub_rn(__fmul_rn(d1, d4), __fmul_rn(d3, d2));
    if (d3 >= 0.0f && d4 <= d3) {
      u = 1.0f; v = 0.0f;
      qx = B.x; qy = B.y; qz = B.z;
    } else if (vc <= 0.0f && d1 >= 0.0f && d3 <= 0.0f) {
      const float s = __fdiv_rn(d1, __fsub_rn(d1, d3));
      u = s; v = 0.0f;
      qx = __fadd_rn(A.x, __fmul_rn(s, abx));
      qy = __fadd_rn(A.y, __fmul_rn(s, aby));
      qz = __fadd_rn(A.z, __fmul_rn(s, abz));
    } else {
      const float cpx = __fsub_rn(px, C.x), cpy = __fsub_rn(py, C.y), cpz = __fsub_rn(pz, C.z);
      const float d5 = cp_dot(abx, aby, abz, cpx, cpy, cpz), d6 = cp_dot(acx, acy, acz, cpx, cpy, cpz);
      const float vb = __fsub_rn(__fmul_rn(d5, d2), __fmul_rn(d1, d6));
      const float va = __fsub_rn(__fmul_rn(d3, d6), __fmul_rn(d5, d4));
      const float e43 = __fsub_rn(d4, d3), e56 = __fsub_rn(d5, d6);
      if (d6 >= 0.0f && d5 <= d6) {
        u = 0.0f; v = 1.0f;
        qx = C.x; qy = C.y; qz = C.z;
      } else if (vb <= 0.0f && d2 >= 0.0f && d6 <= 0.0f) {
        const float s = __fdiv_rn(d2, __fsub_rn(d2, d6));
        u = 0.0f; v = s;
        qx = __fadd_rn(A.x, __fmul_rn(s, acx));
        qy = __fadd_rn(A.y, __fmul_rn(s, acy));
        qz = __fadd_rn(A.z, __fmul_rn(s, acz));
      } else if (va <= 0.0f && e43 >= 0.0f && e56 >= 0.0f) {
        const float s = __fdiv_rn(e43, __fadd_rn(e43, e56));
        u = __fsub_rn(1.0f, s); v = s;
        qx = __fadd_rn(B.x, __fmul_rn(s, __fsub_rn(C.x, B.x)));
        qy = __fadd_rn(B.y, __fmul_rn(s, __fsub_rn(C.y, B.y)));
        qz = __fadd_rn(B.z, __fmul_rn(s, __fsub_rn(C.z, B.z)));
      } else {
        const float r = __fdiv_rn(1.0f, __fadd_rn(__fadd_rn(va, vb), vc));
        float fv = __fmul_rn(vb, r), fw = __fmul_rn(vc, r);
        if (!(fv >= 0.0f)) fv = 0.0f;
        if (!(fw >= 0.0f)) fw = 0.0f;
        const float sum = __fadd_rn(fv, fw);
        if (sum > 1.0f) {
          fv = __fdiv_rn(fv, sum);
          fw = __fdiv_rn(fw, sum);
        }
        u = fv; v = fw;
        qx = __fadd_rn(__fadd_rn(A.x, __fmul_rn(abx, fv)), __fmul_rn(acx, fw));
        qy = __fadd_rn(__fadd_rn(A.y, __fmul_rn(aby, fv)), __fmul_rn(acy, fw));
        qz = __fadd_rn(__fadd_rn(A.z, __fmul_rn(abz, fv)), __fmul_rn(acz, fw));
      }
    }
  }
  const float xx = __fsub_rn(px, qx), xy = __fsub_rn(py, qy), xz = __fsub_rn(pz, qz);
  return cp_dot(xx, xy, xz, xx, xy, xz);
}

// Lower bound on the squared distance from p to any point of the box (see the
// file comment); +inf for an empty box (lo > hi on an axis with infinities)
__device__ __forceinline__ float box_lower(const CpLane &L, float lox, float loy, float loz, float hix, float hiy,
                                           float hiz) {
  const float gx = fmaxf(fmaxf(__fsub_rd(lox, L.px), __fsub_rd(L.px, hix)), 0.0f);
  const float gy = fmaxf(fmaxf(__fsub_rd(loy, L.py), __fsub_rd(L.py, hiy)), 0.0f);
  const float gz = fmaxf(fmaxf(__fsub_rd(loz, L.pz), __fsub_rd(L.pz, hiz)), 0.0f);
  return __fadd_rd(__fadd_rd(__fmul_rd(gx, gx), __fmul_rd(gy, gy)), __fmul_rd(gz, gz));
}

// what a box bound is compared with (see the file comment)
__device__ __forceinline__ float cp_limit(float d2) { return fmaf(d2, 1.0f + 3.814697265625e-06f, 1e-42f); }

// all nine coordinates finite: x * 0 is 0, for infinities and NaN it is NaN
__device__ __forceinline__ bool finite_triangle(float4 p0, float4 p1, float4 p2) {
  float z = p0.x * 0.0f;
  z = fmaf(p0.y, 0.0f, z); z = fmaf(p0.z, 0.0f, z);
  z = fmaf(p1.x, 0.0f, z); z = fmaf(p1.y, 0.0f, z); z = fmaf(p1.z, 0.0f, z);
  z = fmaf(p2.x, 0.0f, z); z = fmaf(p2.y, 0.0f, z); z = fmaf(p2.z, 0.0f, z);
  return z == 0.0f;
}

// triangles [first, first + count): keep the lexicographic minimum of (d2, id)
template <bool STATS>
__device__ __forceinline__ void cp_leaf(const TraceArgs &a, CpLane &L, uint32_t first, uint32_t count,
                                        Counts &cnt) {
  if (STATS) cnt.leaves++;
  for (uint32_t i = first; i < first + count; ++i) {
    if (STATS) cnt.prims++;
    float4 p0, p1, p2;
    uint32_t id;
    if (a.prim_indirect) {
      id = __ldg(a.prim_ids + i);
      uint32_t i0, i1, i2;
      if (a.tri_idx) {
        i0 = __ldg(a.tri_idx + 3 * (size_t)id);
        i1 = __ldg(a.tri_idx + 3 * (size_t)id + 1);
        i2 = __ldg(a.tri_idx + 3 * (size_t)id + 2);
      } else {
        i0 = 3 * id; i1 = i0 + 1; i2 = i0 + 2;
      }
      p0 = ldg4f(a.verts + i0);
      p1 = ldg4f(a.verts + i1);
      p2 = ldg4f(a.verts + i2);
    } else {
      const float4 *q = a.prims + 3 * (size_t)i;
      p0 = ldg4f(q);
      p1 = ldg4f(q + 1);
      p2 = ldg4f(q + 2);
      id = __float_as_uint(p0.w);
    }
    if (!finite_triangle(p0, p1, p2)) continue;
    float u, v;
    const float d2 = cp_triangle(L.px, L.py, L.pz, p0, p1, p2, u, v);
    if (d2 < L.b.d2 || (d2 == L.b.d2 && id < L.b.id)) L.b = CpBest{d2, u, v, id};
  }
}

// next stacked entry whose bound can still hold a closer point
template <class S>
__device__ __forceinline__ uint32_t cp_pop(const CpLane &L, S &st) {
  const float lim = cp_limit(L.b.d2);
  while (!st.empty()) {
    const uint2 e = st.pop();
    if (__uint_as_float(e.y) <= lim) return e.x;
  }
  return kEmptyRef;
}

// Leaf entry: one triangle, as the ray traversal (the counting kernels: all). A
// leaf is one visit, counted with its last triangle.
template <bool STATS, class S>
__device__ __forceinline__ void cp_leaf_wide(const TraceArgs &a, CpLane &L, S &st, Counts &cnt) {
  const uint32_t count = ref_leaf_count(L.cur);
  cp_leaf<STATS>(a, L, ref_leaf_first(L.cur), STATS ? count : 1u, cnt);
  if (!STATS && count > 1u) {
    L.cur += (1u << 5) - (1u << 1);  // ref_leaf(first + 1, count - 1)
    return;
  }
  ++L.steps;
  L.cur = cp_pop(L, st);
}

// Interior node: bound every child box, enter the nearest, stack the others
// (nearest last pushed, so popped first).
template <int W, int PREC, int SOA, int CREF, bool STATS, class S>
__device__ __forceinline__ void cp_node_wide(const TraceArgs &a, CpLane &L, S &st, Counts &cnt) {
  using N = WideNode<W, PREC, SOA, CREF>;
  const uint32_t cur = L.cur;
  ++L.steps;
  if (STATS) cnt.nodes++;
  const uint4 *np = a.nodes + (size_t)ref_node(cur) * (N::kStride / 16);
  uint4 q[N::NQ];
  load_node<N::NQ>(np, q);
  float ox = 0.f, oy = 0.f, oz = 0.f, sx = 0.f, sy = 0.f, sz = 0.f;
  if (N::kGrid) {
    ox = __uint_as_float(q[0].x); oy = __uint_as_float(q[0].y); oz = __uint_as_float(q[0].z);
    sx = __uint_as_float((q[0].w & 0xFFu) << 23);
    sy = __uint_as_float(((q[0].w >> 8) & 0xFFu) << 23);
    sz = __uint_as_float(((q[0].w >> 16) & 0xFFu) << 23);
  }
  const float lim = cp_limit(L.b.d2);
  uint32_t cref[W];
  float clb[W];
  uint32_t base_node = 0, base_prim = 0, leaf_acc = 0;
  if (CREF == REF_INDIRECT) {
    base_node = qword(q, N::kRefOff / 4);
    base_prim = qword(q, N::kRefOff / 4 + 1);
  }
#pragma unroll
  for (int k = 0; k < W; ++k) {
    uint32_t ref;
    if (CREF == REF_DIRECT) {
      ref = qword(q, N::kRefOff / 4 + k);
    } else {
      const uint32_t m = (qword(q, N::kRefOff / 4 + 2 + (k >> 2)) >> ((k & 3) * 8)) & 0xFFu;
      if (m == 0) ref = kEmptyRef;
      else if (m & kMetaInterior) ref = ref_interior(base_node + (m & 0x7Fu));
      else { ref = ref_leaf(base_prim + leaf_acc, m); leaf_acc += m; }
    }
    float lo[3], hi[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      if (PREC == PREC_F32) {
        lo[c] = __uint_as_float(N::raw(q, k, c));
        hi[c] = __uint_as_float(N::raw(q, k, c + 3));
      } else if (PREC == PREC_F16) {
        lo[c] = __half2float(__ushort_as_half((unsigned short)N::raw(q, k, c)));
        hi[c] = __half2float(__ushort_as_half((unsigned short)N::raw(q, k, c + 3)));
      } else {
        const float o = c == 0 ? ox : (c == 1 ? oy : oz), sc = c == 0 ? sx : (c == 1 ? sy : sz);
        lo[c] = fmaf(N::code(q, k, c), sc, o);
        hi[c] = fmaf(N::code(q, k, c + 3), sc, o);
      }
    }
    const float lb = box_lower(L, lo[0], lo[1], lo[2], hi[0], hi[1], hi[2]);
    const bool in = ref != kEmptyRef && lb <= lim;
    cref[k] = in ? ref : kEmptyRef;
    clb[k] = in ? lb : __int_as_float(0x7f800000);
  }
  if (a.ordered == 1) sort_children<W>(clb, cref);
  else if (a.ordered == 2) {
#pragma unroll
    for (int k = W - 1; k > 0; --k) cmpx(clb, cref, k - 1, k);
  }
  uint32_t next = kEmptyRef;
  if (a.ordered && st.sp - st.base + W <= st.cap_sh) {
    // room in shared memory for any node; the nearest child is in slot 0 (one
    // whose bound is +inf may not be: it is then stacked and popped below)
    int sp = st.sp;
#pragma unroll
    for (int k = W - 1; k > 0; --k)
      if (cref[k] != kEmptyRef) st.sh_put(st.slot(sp++), make_uint2(cref[k], __float_as_uint(clb[k])));
    st.sp = sp;
    next = cref[0];
  } else {
    float next_lb = 0.f;
#pragma unroll
    for (int k = W - 1; k >= 0; --k) {
      if (cref[k] == kEmptyRef) continue;
      if (next != kEmptyRef && !st.push(next, next_lb)) { L.err = kErrStack; L.cur = kEmptyRef; return; }
      next = cref[k];
      next_lb = clb[k];
    }
  }
  L.cur = next != kEmptyRef ? next : cp_pop(L, st);
}

// Next stacked node of an own-box query, with its reference.
template <int PREC, int SOA, class S>
__device__ __forceinline__ void cp_bin_pop(const TraceArgs &a, CpLane &L, S &st) {
  L.cur = cp_pop(L, st);
  if (L.cur != kEmptyRef) own_ref<PREC, SOA>(a, L.cur, L.count, L.field);
}

// Leaf of an own-box query: one triangle (the counting kernels: all).
template <int PREC, int SOA, bool STATS, class S>
__device__ __forceinline__ void cp_leaf_bin(const TraceArgs &a, CpLane &L, S &st, Counts &cnt) {
  if (STATS) cnt.nodes++;
  cp_leaf<STATS>(a, L, L.field, STATS ? L.count : 1u, cnt);
  if (!STATS && --L.count > 0) {
    ++L.field;
    return;
  }
  ++L.steps;
  cp_bin_pop<PREC, SOA>(a, L, st);
}

// Own-box interior node (the entered node's box was bounded by its parent):
// bounds both children's boxes (the paper's children sorting), enters the nearer
// and stacks the other.
template <int PREC, int SOA, int CREF, bool STATS, class S>
__device__ __forceinline__ void cp_node_bin(const TraceArgs &a, CpLane &L, S &st, Counts &cnt) {
  ++L.steps;
  if (STATS) cnt.nodes++;
  const uint32_t l = CREF == REF_DIRECT ? L.cur + 1 : L.field;
  const uint32_t r = CREF == REF_DIRECT ? L.cur + L.field : L.field + 1;
  float llo[3], lhi[3], rlo[3], rhi[3];
  uint32_t lc, lf, rc, rf;
  own_node<PREC, SOA>(a, l, llo, lhi, lc, lf);
  own_node<PREC, SOA>(a, r, rlo, rhi, rc, rf);
  const float lim = cp_limit(L.b.d2);
  const float bl = box_lower(L, llo[0], llo[1], llo[2], lhi[0], lhi[1], lhi[2]);
  const float br = box_lower(L, rlo[0], rlo[1], rlo[2], rhi[0], rhi[1], rhi[2]);
  const bool inl = bl <= lim, inr = br <= lim;
  if (!inl && !inr) {
    cp_bin_pop<PREC, SOA>(a, L, st);
    return;
  }
  const bool right = inr && (!inl || (a.ordered && br < bl));
  if (inl && inr && !st.push(right ? l : r, right ? bl : br)) { L.err = kErrStack; L.cur = kEmptyRef; return; }
  L.cur = right ? r : l;
  L.count = right ? rc : lc;
  L.field = right ? rf : lf;
}

// Closest point queries as a query of refill_loop. Random neighbours share little of
// their paths: in batches of 32 a warp had 4 of its lanes active. Idle lanes are
// refilled, except while a warp's points go together, and a leaf runs triangle by
// triangle; 1 M random points around 1.4 M triangles, before and
// after: bvh4 f32 5.90 -> 3.65 ms, bvh8 f16 7.47 -> 5.48, bvh2 q16 6.89 -> 4.47; with
// nodes and triangles in one step (node_then_leaf) 3.33, 4.53 and 3.90.
template <bool OWN, int W, int PREC, int SOA, int CREF, bool STATS, class S>
struct PointQuery {
  S &st;
  CpLane L;
  Counts cnt;
  uint32_t n_pts = 0;
  __device__ __forceinline__ explicit PointQuery(S &stack) : st(stack) {}
  __device__ __forceinline__ void idle() { L.cur = kEmptyRef; }
  __device__ __forceinline__ bool busy() const { return L.cur != kEmptyRef; }
  __device__ __forceinline__ void start(const TraceArgs &a, unsigned long long rid) {
    const float4 pt = ldg4f(a.rays + rid);
    L.rid = rid;
    L.px = pt.x; L.py = pt.y; L.pz = pt.z;
    L.b = CpBest{pt.w, 0.f, 0.f, SCION_PRIM_MISS};
    L.steps = 0;
    L.err = 0;
    st.reset();
    // a point that is not finite, or a radius that is not >= 0, finds nothing
    const bool live = isfinite(pt.x) && isfinite(pt.y) && isfinite(pt.z) && pt.w >= 0.0f;
    if constexpr (OWN) {
      L.cur = live && a.n_nodes > 0 ? 0u : kEmptyRef;
      if (L.cur == 0u) own_ref<PREC, SOA>(a, 0u, L.count, L.field);
    } else {
      L.cur = live ? a.root_ref : kEmptyRef;
    }
    if (STATS) n_pts++;
  }
  __device__ __forceinline__ void step(const TraceArgs &a) {
    if constexpr (OWN) {
      node_then_leaf<2>(
          L, [&] { return L.count > 0; }, [&] { cp_node_bin<PREC, SOA, CREF, STATS>(a, L, st, cnt); },
          [&] { cp_leaf_bin<PREC, SOA, STATS>(a, L, st, cnt); });
    } else {
      node_then_leaf<W <= 4 ? 2 : 1>(
          L, [&] { return !ref_is_interior(L.cur); }, [&] { cp_node_wide<W, PREC, SOA, CREF, STATS>(a, L, st, cnt); },
          [&] { cp_leaf_wide<STATS>(a, L, st, cnt); });
    }
    if (L.steps > a.max_steps) {
      L.err = kErrIter;
      L.cur = kEmptyRef;
    }
  }
  __device__ __forceinline__ void finish(const TraceArgs &a) {
    if (L.err) {
      atomicCAS(a.status, 0u, L.err);
      L.b = CpBest{__int_as_float(0x7f800000), 0.f, 0.f, SCION_PRIM_ERROR};
    }
    if (L.b.id == SCION_PRIM_MISS) L.b.d2 = __int_as_float(0x7f800000);
    static_cast<uint4 *>(a.out)[L.rid] =
        make_uint4(__float_as_uint(L.b.d2), __float_as_uint(L.b.u), __float_as_uint(L.b.v), L.b.id);
  }
  __device__ __forceinline__ void report(const TraceArgs &a) const {
    if (!STATS) return;
    atomicAdd(a.stats + 0, (unsigned long long)cnt.nodes);
    atomicAdd(a.stats + 1, (unsigned long long)cnt.leaves);
    atomicAdd(a.stats + 2, (unsigned long long)cnt.prims);
    atomicAdd(a.stats + 3, (unsigned long long)n_pts);
  }
};

template <bool OWN, int W, int PREC, int SOA, int CREF, bool STATS>
__device__ __forceinline__ void cpq_kernel_body(const TraceArgs &a) {
  extern __shared__ uint2 smem_stack[];
  StackFor<OWN, PREC, W, false, 0> st;
  StackTail<false> tail;
  st.attach(tail);
  st.columns(smem_stack, a.smem_stack);
  st.reset();
  PointQuery<OWN, W, PREC, SOA, CREF, STATS, decltype(st)> q(st);
  trace_loop<true>(a, q);
  q.report(a);
}

}  // namespace scion
