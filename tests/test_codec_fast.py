"""The FP32 box codecs of the device encoders (codec_fast.h) give the bytes of
the double-precision codecs (codec.h): both compiled for the host and compared
on random and degenerate boxes (flat, dyadic, at zero, scales from denormal
numbers to the largest floats)."""
import os
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2511_15028_gb300", "csrc")

SOURCE = r"""
#include <cstdio>
#include <random>
#include "codec_fast.h"
using namespace scion;
static std::mt19937_64 rng(1);
static double U(double a, double b) { return a + (b - a) * (rng() >> 11) * (1.0 / 9007199254740992.0); }

// a u8 / u16 node as the device encoder composes it
template <int W, int P>
static int node(const Box3 *ex, const bool *live, uint32_t soa, uint8_t *b) {
  const uint32_t qmax = P == PREC_U8 ? 255 : 65535;
  Box3 cb[W], m;
  bool any = false;
  for (int a = 0; a < 3; ++a) m.lo[a] = INFINITY, m.hi[a] = -INFINITY;
  for (int k = 0; k < W; ++k)
    if (live[k]) {
      any = true;
      cb[k] = padded_fast(ex[k]);
      for (int a = 0; a < 3; ++a) m.lo[a] = fminf(m.lo[a], cb[k].lo[a]), m.hi[a] = fmaxf(m.hi[a], cb[k].hi[a]);
    }
  if (!any)
    for (int a = 0; a < 3; ++a) m.lo[a] = m.hi[a] = 0;
  const PadPair g = pad_pair(m);
  const Box3 fr = padded_fast(m);
  int bad = 0;
  for (int a = 0; a < 3; ++a) {
    const FrameAxis f = frame_axis(fr, a, qmax);
    memcpy(b + 4 * a, &f.origin, 4);
    b[12 + a] = (uint8_t)(f.e + 127);
    for (int k = 0; k < W; ++k) {
      uint32_t lo = qmax, hi = 0;
      if (live[k] && !frame_codes(cb[k].lo[a], cb[k].hi[a], m, g, f, qmax, &lo, &hi)) bad |= 4;
      memcpy(b + wide_box_offset(W, P, soa, k, a), &lo, P == PREC_U8 ? 1 : 2);
      memcpy(b + wide_box_offset(W, P, soa, k, 3 + a), &hi, P == PREC_U8 ? 1 : 2);
    }
  }
  return bad;
}
template <int W, int P>
static long differs(const Box3 *v, int n, uint32_t soa) {
  uint8_t a[512] = {0}, b[512] = {0};
  Box3 ex[8];
  bool live[8];
  for (int k = 0; k < W; ++k) {
    ex[k] = k < n ? v[k] : Box3{{9, 9, 9}, {8, 8, 8}};
    live[k] = !box_is_empty(ex[k]);
  }
  const int ra = encode_wide_boxes(W, P, soa, ex, n < W ? n : W, a), rb = node<W, P>(ex, live, soa, b);
  return ra != rb || memcmp(a, b, 512);
}

int main() {
  long pad = 0, grid = 0, wide = 0;
  for (int it = 0; it < 60000; ++it) {
    const int mode = rng() % 12, n = 1 + rng() % 8;
    double sc = mode == 2 ? 1e-3 : (mode == 3 ? 1e4 : 1);
    if (mode == 1) sc = std::pow(10, U(-30, 30));
    if (mode == 9) sc = std::pow(2, U(98, 127.99));  // extents to twice the largest float
    if (mode == 10) sc = std::pow(2, U(-149, -100));
    if (mode == 11) sc = std::ldexp(1.0, 100 + (int)(rng() % 28));
    Box3 v[8];
    double c[3];
    for (double &x : c) x = mode == 4 ? 0 : U(-1, 1) * sc;
    for (int k = 0; k < 8; ++k) {
      for (int a = 0; a < 3; ++a) {
        double w = std::pow(10, U(-6, 0)) * sc;
        if (mode == 5) w = 0;
        if (mode == 6) w = std::floor(U(0, 64)) / 64;
        double l = c[a] + U(-1, 1) * w;
        if (mode == 6) l = std::floor(U(-64, 64)) / 32;
        if (mode == 7) l = std::floor(U(-8, 8));
        if (mode == 8 && rng() % 3 == 0) l = 0;
        v[k].lo[a] = fminf(fmaxf((float)l, -3.4028235e38f), 3.4028235e38f);
        v[k].hi[a] = fminf(fmaxf((float)(l + w), v[k].lo[a]), 3.4028235e38f);
      }
      if (rng() % 40 == 0) v[k].lo[0] = INFINITY, v[k].hi[0] = -INFINITY;
      if (box_is_empty(v[k])) continue;
      const Box3 p = padded(v[k]), q = padded_fast(v[k]);
      pad += memcmp(&p, &q, sizeof p) != 0;
      const float wlo = (float)(v[k].lo[0] - U(0, 2) * sc), whi = (float)(v[k].hi[0] + U(0, 2) * sc);
      const float st = q16_step(wlo, whi);
      uint32_t a1, b1, a2, b2;
      const bool o1 = q16_codes(v[k].lo[0], v[k].hi[0], st, wlo, &a1, &b1);
      const bool o2 = q16_codes_fast(v[k].lo[0], v[k].hi[0], st, wlo, reciprocal_pair(st), &a2, &b2);
      grid += o1 != o2 || a1 != a2 || b1 != b2;
    }
    const uint32_t soa = rng() & 1;
    wide += differs<2, PREC_U8>(v, n, soa) + differs<4, PREC_U8>(v, n, soa) + differs<8, PREC_U8>(v, n, soa) +
            differs<2, PREC_U16>(v, n, soa) + differs<4, PREC_U16>(v, n, soa) + differs<8, PREC_U16>(v, n, soa);
  }
  std::printf("%ld %ld %ld\n", pad, grid, wide);
}
"""


@pytest.mark.parametrize("opt", ["-O0", "-O2"])
def test_fast_codecs_equal_the_double_precision_codecs(tmp_path, opt):
    src = tmp_path / "codec.cpp"
    src.write_text(SOURCE)
    exe = tmp_path / "codec"
    subprocess.run(["g++", opt, "-std=c++17", "-ffp-contract=off", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True, timeout=300).stdout.split()
    assert out == ["0", "0", "0"], f"padded boxes, q16 codes, u8/u16 nodes that differ: {out}"
