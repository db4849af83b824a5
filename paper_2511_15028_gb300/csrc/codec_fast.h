// The box codecs of codec.h for the refit, byte for byte the same codes without
// its double-precision arithmetic (FP64 has a small fraction of the FP32 rate on
// this part: with codec.h the encoder was bound by it, 0.8 ms for 1.4 M
// triangles).
//
// codec.h computes pads, frames and codes in double and rounds them to float
// or to an integer in a given direction. Here such a value is carried as an
// unevaluated sum of two floats (error-free transformations: TwoSum by Knuth,
// products by one fma), about 2^-46 accurate. The direction of the rounding
// is then certain unless the value lies within that error of a float or an
// integer; those few cases, and ranges where the pairs could underflow or
// overflow, are computed as codec.h does. Compiled for host and device.
#pragma once

#include "codec.h"

#if defined(__CUDACC__)
#include <cuda_fp16.h>
#endif

#if defined(__CUDACC__)
#define SCION_SLOW __host__ __device__ __noinline__ inline  // rare: kept out of line
#define SCION_UNROLL _Pragma("unroll")
#else
#define SCION_SLOW inline
#define SCION_UNROLL
#endif

namespace scion {

struct FPair {
  float hi, lo;
};
SCION_HD FPair two_sum(float a, float b) {
  const float s = a + b, t = s - a;
  return {s, (a - (s - t)) + (b - t)};
}
SCION_HD uint32_t float_bits(float x) {
  uint32_t u;
  memcpy(&u, &x, 4);
  return u;
}
SCION_HD float bits_float(uint32_t u) {
  float x;
  memcpy(&x, &u, 4);
  return x;
}
// the floats next to a finite x
SCION_HD float next_below(float x) {
  const uint32_t u = float_bits(x);
  return bits_float(x == 0.0f ? 0x80000001u : ((u >> 31) ? u + 1u : u - 1u));
}
SCION_HD float next_above(float x) { return -next_below(-x); }
// x 2^e for a power of two within the exponent range of normal floats
SCION_HD float pow2f(int e) { return bits_float((uint32_t)(e + 127) << 23); }

// The pad of `padded` (2^-20 (largest extent + largest |coordinate|)) as a pair.
struct PadPair {
  float hi, lo;
  bool usable;  // the pair holds it to 2^-46
  bool exact;   // the pair is exactly it
};
SCION_HD PadPair pad_pair(const Box3 &b) {
  FPair ext{0.0f, 0.0f};
  float mag = 0.0f;
  SCION_UNROLL
  for (int a = 0; a < 3; ++a) {
    const FPair d = two_sum(b.hi[a], -b.lo[a]);
    if (d.hi > ext.hi || (d.hi == ext.hi && d.lo > ext.lo)) ext = d;
    mag = fmaxf(mag, fmaxf(fabsf(b.lo[a]), fabsf(b.hi[a])));
  }
  const FPair s = two_sum(ext.hi, mag);
  const float low = s.lo + ext.lo;
  const float hi = s.hi + low, lo = low - (hi - s.hi);
  PadPair p;
  p.hi = hi * 9.5367431640625e-07f;  // 2^-20
  p.lo = lo * 9.5367431640625e-07f;
  p.usable = hi > 1e-16f && hi < 1e30f;  // neither part leaves the normal range
  p.exact = s.lo == 0.0f || ext.lo == 0.0f;
  return p;
}
// The same pad in double.
SCION_HD double pad_double(const Box3 &b) {
  double ext = 0.0, mag = 0.0;
  for (int a = 0; a < 3; ++a) {
    ext = fmax(ext, (double)b.hi[a] - (double)b.lo[a]);
    mag = fmax(mag, fmax(fabs((double)b.lo[a]), fabs((double)b.hi[a])));
  }
  return ldexp(ext + mag, -20);
}
// x - pad rounded to float toward -inf as round_down_f32((double)x - pad)
// rounds it; false if the pair cannot tell.
SCION_HD bool sub_pad_down(float x, const PadPair &p, float *out) {
  const FPair d = two_sum(x, -p.hi);
  const float r = d.lo - p.lo;  // x - pad = d.hi + r
  if (r == 0.0f) {
    *out = d.hi;
    return p.exact && p.lo == 0.0f;
  }
  const float unsure = fmaxf(fabsf(d.hi), p.hi) * 5.684341886080802e-14f;  // 2^-44
  if (r > 0.0f) {
    *out = d.hi;
    return r > unsure && r < (next_above(d.hi) - d.hi) - unsure;
  }
  const float g = next_below(d.hi);
  *out = g;
  return -r > unsure && (d.hi - g) + r > unsure;
}
SCION_SLOW Box3 padded_slow(const Box3 &b) { return padded(b); }
// padded(b), the same floats.
SCION_HD Box3 padded_fast(const Box3 &b) {
  const PadPair p = pad_pair(b);
  Box3 o;
  bool sure = p.usable;
  if (sure) {
    SCION_UNROLL
    for (int a = 0; a < 3; ++a) {
      float hi;
      sure &= sub_pad_down(b.lo[a], p, &o.lo[a]);
      sure &= sub_pad_down(-b.hi[a], p, &hi);
      o.hi[a] = -hi;
    }
  }
  return sure ? o : padded_slow(b);
}

// ------------------------------------------------------------ world grid
// floor and ceil of (x - wlo) / step as q16_codes takes them; inv: 1 / step as
// a pair.
SCION_HD FPair reciprocal_pair(float step) {
  if (!(step > 0.0f)) return {0.0f, 0.0f};
  const double r = 1.0 / (double)step;
  const float hi = (float)r;
  return {hi, (float)(r - (double)hi)};
}
SCION_SLOW double q16_floor_slow(float x, float wlo, float step, bool up) {
  const double q = ((double)x - (double)wlo) / (double)step;
  return up ? ceil(q) : floor(q);
}
SCION_HD uint32_t q16_floor(float x, float wlo, float step, const FPair &inv, bool up) {
  const FPair d = two_sum(x, -wlo);
  const float p = d.hi * inv.hi;
  const float e = fmaf(d.hi, inv.hi, -p) + (d.hi * inv.lo + d.lo * inv.hi);
  const float f = floorf(p), frac = (p - f) + e;  // the quotient is f + frac
  double v;
  if (frac > 1e-5f && frac < 1.0f - 1e-5f) v = (double)(up ? f + 1.0f : f);
  else v = q16_floor_slow(x, wlo, step, up);
  return clamp_code(v, kQ16Max);
}
SCION_HD bool q16_codes_fast(float lo, float hi, float step, float wlo, const FPair &inv, uint32_t *qlo,
                             uint32_t *qhi) {
  uint32_t a = 0, b = 0;
  if (step > 0.0f) {
    a = q16_floor(lo, wlo, step, inv, false);
    b = q16_floor(hi, wlo, step, inv, true);
  }
  while (a > 0 && q16_decode(a, step, wlo) > lo) --a;
  while (b < kQ16Max && q16_decode(b, step, wlo) < hi) ++b;
  *qlo = a;
  *qhi = b;
  return q16_decode(a, step, wlo) <= lo && q16_decode(b, step, wlo) >= hi;
}
#if defined(__CUDACC__)
// eq10 in directed FP32 instructions, which is what codec.h emulates
__device__ __forceinline__ uint32_t clamp_code_f(float v, uint32_t qmax) {
  return v > 0.0f ? (v >= (float)qmax ? qmax : (uint32_t)v) : 0u;
}
__device__ __forceinline__ bool eq10_codes_fast(float lo, float hi, float bin, float bins_inv, float wlo, float whi,
                                                uint32_t *qlo, uint32_t *qhi) {
  uint32_t a = clamp_code_f(floorf(__fmul_rd(__fsub_rd(lo, wlo), bins_inv)), kEq10Max);
  uint32_t b = clamp_code_f(floorf(__fmul_rd(__fsub_rd(whi, hi), bins_inv)), kEq10Max);
  while (a > 0 && __fmaf_rd((float)a, bin, wlo) > lo) --a;
  while (b > 0 && __fmaf_ru(-(float)b, bin, whi) < hi) --b;
  *qlo = a;
  *qhi = b;
  return __fmaf_rd((float)a, bin, wlo) <= lo && __fmaf_ru(-(float)b, bin, whi) >= hi;
}

// encode_own_box, the same bytes; inv: reciprocal_pair of the q16 steps.
__device__ inline bool encode_own_box_fast(uint32_t prec, const Box3 &exact, const float *frame,
                                           const float *bins_inv, const FPair *inv, uint32_t (&w)[6]) {
  const bool empty = box_is_empty(exact);
  const Box3 b = empty ? exact : padded_fast(exact);
  if (prec == PREC_F32) {
    for (int a = 0; a < 3; ++a) {
      w[a] = float_bits(empty ? INFINITY : b.lo[a]);
      w[3 + a] = float_bits(empty ? -INFINITY : b.hi[a]);
    }
    return true;
  }
  bool ok = true;
  uint32_t qlo[3], qhi[3];
  for (int a = 0; a < 3; ++a) {
    if (empty) {
      qlo[a] = prec == PREC_Q16 ? kQ16Max : kEq10Max;
      qhi[a] = prec == PREC_Q16 ? 0u : kEq10Max;
      continue;
    }
    ok &= prec == PREC_Q16 ? q16_codes_fast(b.lo[a], b.hi[a], frame[3 + a], frame[a], inv[a], &qlo[a], &qhi[a])
                           : eq10_codes_fast(b.lo[a], b.hi[a], frame[6 + a], bins_inv[a], frame[a], frame[3 + a],
                                             &qlo[a], &qhi[a]);
  }
  if (prec == PREC_Q16) {
    w[0] = qlo[0] | qlo[1] << 16;
    w[1] = qlo[2] | qhi[0] << 16;
    w[2] = qhi[1] | qhi[2] << 16;
  } else {
    w[0] = eq10_pack(qlo[0], qlo[1], qlo[2]);
    w[1] = eq10_pack(qhi[0], qhi[1], qhi[2]);
  }
  return ok;
}
// words that encode_own_box_fast fills
__device__ __forceinline__ int own_box_words(uint32_t prec) { return prec == PREC_F32 ? 6 : (prec == PREC_Q16 ? 3 : 2); }
#endif

// ------------------------------------------------------------ u8 / u16 frames
// Smallest e >= -126 with qmax 2^e >= span, span = fhi - origin > 0 (the loop of
// encode_wide_boxes ends there too).
SCION_SLOW int frame_exponent_slow(float fhi, float origin, uint32_t qmax) {
  const double span = (double)fhi - (double)origin;
  int e = -126;
  while (e < 127 && ldexp((double)qmax, e) < span) ++e;
  return e;
}
SCION_HD int frame_exponent(float fhi, float origin, uint32_t qmax) {
  const FPair s = two_sum(fhi, -origin);
  if (!(s.hi > 0.0f)) return -126;
  // below, every qmax 2^e up to the one that is returned is a finite float
  if (!(s.hi < 1e33f)) return frame_exponent_slow(fhi, origin, qmax);
  const int es = (int)((float_bits(s.hi) >> 23) & 255u) - 127;  // 2^es <= s.hi < 2^(es + 1)
  int e = es - (qmax == 255u ? 8 : 16);
  if (e < -126) e = -126;
  while (true) {
    // qmax 2^e is a float; its equality with the leading part is left to the
    // trailing part (rounded away in double only where it is below 2^-52 of the
    // span)
    const float reach = (float)qmax * pow2f(e);
    if (reach > s.hi || (reach == s.hi && s.lo <= s.hi * 1.1102230246251565e-16f)) break;
    ++e;
  }
  return e;
}
// floor((x - g - origin) / 2^e) for the pad g, as encode_wide_boxes computes it;
// false if the pair cannot tell.
SCION_HD bool frame_floor(float x, const PadPair &g, float origin, int e, float *out) {
  const FPair d = two_sum(x, -origin), s = two_sum(d.hi, -g.hi);
  const float r = s.lo + (d.lo - g.lo);
  // scaled by 2^-e: exact while the parts stay in the normal range
  if (e < -60 || e > 60) return false;
  const float k = pow2f(-e), v = s.hi * k, f = floorf(v), frac = (v - f) + r * k;
  *out = f;
  return frac > 1e-6f && frac < 1.0f - 1e-6f;
}

// Code targets of a child's interval on one axis, in double: the first codes
// (fl, fh) and the floats that decoded codes are compared with.
struct FrameCodes {
  float fl, fh, tlo, thi;
};
SCION_SLOW FrameCodes frame_codes_slow(float blo, float bhi, const Box3 &merged, float origin, int e, float qmax) {
  const double g = pad_double(merged);
  const double lo = (double)blo - g, hi = (double)bhi + g;
  const double inv = ldexp(1.0, -e);  // division by a power of two
  FrameCodes c;
  c.fl = (float)fmin((double)qmax, fmax(0.0, floor((lo - (double)origin) * inv)));
  c.fh = (float)fmin((double)qmax, fmax(0.0, ceil((hi - (double)origin) * inv)));
  c.tlo = round_down_f32(lo);
  c.thi = round_up_f32(hi);
  return c;
}

// One axis of a u8 / u16 node's frame: the origin and scale 2^e for the merged
// child box grown by its own pad (fr = padded_fast(merged)).
struct FrameAxis {
  float origin, scale;
  int e;
};
SCION_HD FrameAxis frame_axis(const Box3 &fr, int a, uint32_t qmax) {
  FrameAxis f;
  f.origin = fr.lo[a];
  f.e = frame_exponent(fr.hi[a], fr.lo[a], qmax);
  f.scale = f.e >= -126 ? pow2f(f.e) : 0.0f;
  return f;
}
// Codes of a child's padded interval [lo, hi] on one axis as encode_wide_boxes
// finds them; g: the pad of the merged box. False if they cannot enclose it.
SCION_HD bool frame_codes(float lo, float hi, const Box3 &merged, const PadPair &g, const FrameAxis &f, uint32_t qmax,
                          uint32_t *qlo, uint32_t *qhi) {
  FrameCodes c;
  bool sure = g.usable && frame_floor(lo, g, f.origin, f.e, &c.fl) && sub_pad_down(lo, g, &c.tlo);
  // ceil(hi + g - origin) = floor + 1 off the integers; hi + g = -(-hi - g)
  const PadPair ng{-g.hi, -g.lo, true, g.exact};
  sure = sure && frame_floor(hi, ng, f.origin, f.e, &c.fh) && sub_pad_down(-hi, g, &c.thi);
  c.fh += 1.0f;
  c.thi = -c.thi;
  if (!sure) c = frame_codes_slow(lo, hi, merged, f.origin, f.e, (float)qmax);
  // a decoded float is above (below) the exact target iff it is above (below)
  // the target rounded down (up) to float
  uint32_t a = (uint32_t)fminf((float)qmax, fmaxf(0.0f, c.fl)), b = (uint32_t)fminf((float)qmax, fmaxf(0.0f, c.fh));
  while (a > 0 && u8_decode(a, f.scale, f.origin) > c.tlo) --a;
  while (b < qmax && u8_decode(b, f.scale, f.origin) < c.thi) ++b;
  *qlo = a;
  *qhi = b;
  return u8_decode(a, f.scale, f.origin) <= c.tlo && u8_decode(b, f.scale, f.origin) >= c.thi;
}

#if defined(__CUDACC__)
// words of a wide node's header and boxes
template <int W, int PREC>
__host__ __device__ constexpr int wide_box_words() {
  return ((PREC == PREC_U8 || PREC == PREC_U16 ? 16 : 0) + W * 6 * (PREC == PREC_F32 ? 4 : (PREC == PREC_U8 ? 1 : 2))) / 4;
}

// Header and boxes of a wide node as encode_wide_boxes writes them, by W
// neighbouring lanes of a warp, lane k of them with the exact box of child k
// (live: the slot has a child and its box is not empty); all 32 lanes call. p:
// the node's bytes, in shared memory. Returns encode_wide_boxes's flags for
// the lane's child. A lane per child keeps 8 children of a node from being one
// thread's registers (149 of them) and dependent work: 219 -> 112 us for
// the 0.2 M 8-wide u8 nodes of 1.4 M triangles.
template <int W, int PREC>
__device__ __forceinline__ int encode_wide_lane(const Box3 &exact, bool live, uint32_t k, uint32_t soa, uint8_t *p) {
  int bad = 0;
  const Box3 b = live ? padded_fast(exact) : exact;
  if constexpr (PREC == PREC_F32 || PREC == PREC_F16) {
#pragma unroll
    for (int c = 0; c < 6; ++c) {
      const uint32_t off = wide_box_offset(W, PREC, soa, k, c);
      const float v = live ? (c < 3 ? b.lo[c % 3] : b.hi[c % 3]) : (c < 3 ? INFINITY : -INFINITY);
      if constexpr (PREC == PREC_F32) {
        *reinterpret_cast<float *>(p + off) = v;
      } else {
        const __half h = c < 3 ? __float2half_rd(v) : __float2half_ru(v);
        const float dec = __half2float(h);
        if (live && !(c < 3 ? dec <= v : dec >= v)) bad = 2;
        *reinterpret_cast<uint16_t *>(p + off) = __half_as_ushort(h);
      }
    }
  } else {
    constexpr uint32_t qmax = PREC == PREC_U8 ? 255u : 65535u;
    Box3 m;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      m.lo[a] = live ? b.lo[a] : INFINITY;
      m.hi[a] = live ? b.hi[a] : -INFINITY;
#pragma unroll
      for (int o = 1; o < W; o <<= 1) {
        m.lo[a] = fminf(m.lo[a], __shfl_xor_sync(0xFFFFFFFFu, m.lo[a], o));
        m.hi[a] = fmaxf(m.hi[a], __shfl_xor_sync(0xFFFFFFFFu, m.hi[a], o));
      }
    }
    if (!(m.lo[0] <= m.hi[0]))  // no live child
      for (int a = 0; a < 3; ++a) m.lo[a] = m.hi[a] = 0.0f;
    const PadPair g = pad_pair(m);
    const Box3 fr = padded_fast(m);
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      const FrameAxis f = frame_axis(fr, a, qmax);
      if (k == 0) {
        reinterpret_cast<float *>(p)[a] = f.origin;
        p[12 + a] = (uint8_t)(f.e + 127);
      }
      uint32_t qlo = qmax, qhi = 0;
      if (live && !frame_codes(b.lo[a], b.hi[a], m, g, f, qmax, &qlo, &qhi)) bad = 4;
      const uint32_t lo_off = wide_box_offset(W, PREC, soa, k, a), hi_off = wide_box_offset(W, PREC, soa, k, 3 + a);
      if constexpr (PREC == PREC_U8) {
        p[lo_off] = (uint8_t)qlo;
        p[hi_off] = (uint8_t)qhi;
      } else {
        *reinterpret_cast<uint16_t *>(p + lo_off) = (uint16_t)qlo;
        *reinterpret_cast<uint16_t *>(p + hi_off) = (uint16_t)qhi;
      }
    }
    if (k == 0) p[15] = 0;  // the header's spare byte
  }
  return bad;
}
#endif

}  // namespace scion
