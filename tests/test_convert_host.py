"""The integer conversions between FP64 and double-float pairs (convert.cuh)
against the plain ones, bit for bit: compiled for the host, with the few device
functions that the header uses written out in C++.  Pairs with every kind of
neighbourhood (the high word a power of two above all, where the sum may fall
into the binade below), doubles of both signs with and without a low word."""
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2508_05400_gb300", "csrc")

SRC = r"""
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstring>
#include <random>
#define __device__
#define __forceinline__ inline
struct float2 { float x, y; };
static float2 make_float2(float x, float y) { return {x, y}; }
template <class A, class B> static A cast(B b) { A a; std::memcpy(&a, &b, sizeof a); return a; }
static unsigned __float_as_uint(float f) { return cast<unsigned>(f); }
static float __uint_as_float(unsigned u) { return cast<float>(u); }
static float __int_as_float(int u) { return cast<float>(u); }
static int __float2int_rn(float f) {   // the hardware saturates, NaN gives 0
  if (f != f) return 0;
  if (f >= 2147483648.f) return 0x7FFFFFFF;
  if (f < -2147483648.f) return (int)0x80000000u;
  return (int)std::nearbyint(f);
}
static float __int2float_rn(int i) { return (float)i; }
static float __double2float_rn(double d) { return (float)d; }
static double __hiloint2double(int h, int l) { return cast<double>(((uint64_t)(uint32_t)h << 32) | (uint32_t)l); }
static int __double2hiint(double d) { return (int)(cast<uint64_t>(d) >> 32); }
static int __double2loint(double d) { return (int)(uint32_t)cast<uint64_t>(d); }
#include "convert_nocuda.cuh"
static bool same(double a, double b) { return cast<uint64_t>(a) == cast<uint64_t>(b) || (a != a && b != b); }
static bool same(float a, float b) { return cast<unsigned>(a) == cast<unsigned>(b) || (a != a && b != b); }
int main(int, char** argv) {
  std::mt19937_64 g(12345);
  long bad = 0;
  const bool to = argv[1][0] == 't';
  for (long t = 0; t < 3000000; ++t) {
    const uint64_t r = g(), q = g();
    if (to) {
      // hi: random, a power of two, or next to one; lo within half a unit of hi's last place (a few beyond)
      unsigned h = (unsigned)r;
      if (t % 3 == 0) h &= 0xFF800000u;
      if (t % 3 == 1) h = (h & 0xFF800000u) + (unsigned)(r >> 62) - 1u;
      const float hi = __uint_as_float(h);
      float lo;
      if (t % 7 == 0) lo = __uint_as_float((unsigned)q);
      else lo = (float)std::ldexp((double)(int64_t)q, -63 - 24 - (int)(q % 40) + (std::isfinite(hi) && hi != 0 ? std::ilogb(hi) : 0));
      bad += !same(rks::df_to_double(make_float2(hi, lo)), (double)hi + (double)lo);
      if (t % 5 == 0) bad += !same(rks::df_to_double(make_float2(hi, 0.f)), (double)hi + 0.0);
    } else {
      double x = cast<double>(r);
      if (t % 2) x = std::ldexp((double)(int64_t)r, -63 + (int)(q % 280) - 140);
      if (t % 8 == 1) x = (double)(float)x;                       // no low word
      if (t % 8 == 3) x = cast<double>(cast<uint64_t>(x) & ~0x1FFFFFFFull | 0x10000000ull);   // halfway
      if (t % 1000 == 0) x = t % 2000 ? 0.0 : -0.0;
      const float h = (float)x, l = (float)(x - (double)h);
      const float2 v = rks::df_from_double(x);
      bad += !same(v.x, h) || !same(v.y, l);
    }
  }
  std::printf("%ld\n", bad);
  return 0;
}
"""


@pytest.mark.parametrize("way", ["to_double", "from_double"])
def test_conversions_give_the_plain_bits(tmp_path, way):
    hdr = open(os.path.join(CSRC, "convert.cuh")).read()
    (tmp_path / "convert_nocuda.cuh").write_text(hdr.replace("#include <cuda_runtime.h>", ""))
    (tmp_path / "t.cpp").write_text(SRC)
    exe = str(tmp_path / "t")
    subprocess.run(["g++", "-O2", "-ffp-contract=off", "-std=c++17", "-o", exe, str(tmp_path / "t.cpp")], check=True)
    out = subprocess.run([exe, way], capture_output=True, text=True, check=True).stdout
    assert int(out) == 0
