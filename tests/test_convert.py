"""The FP64 <-> FP32 conversions on integer operations (csrc/rt_convert.cuh),
compiled for the host, give the bits of the hardware's conversions: random bit
patterns, every exponent with the mantissas around its rounding points, ties, the
ends of the FP32 range, subnormal numbers, zeros, infinities; NaN stays NaN."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2110_11873_gb300", "csrc")

HOST = r"""
#include <cstdint>
#include <cstdio>
#include <cstring>
#define __device__
#define __forceinline__ inline
static inline uint64_t bits(double x) { uint64_t u; memcpy(&u, &x, 8); return u; }
static inline int __double2hiint(double x) { return (int)(bits(x) >> 32); }
static inline int __double2loint(double x) { return (int)bits(x); }
static inline double __hiloint2double(int h, int l) {
  const uint64_t u = (uint64_t)(uint32_t)h << 32 | (uint32_t)l; double x; memcpy(&x, &u, 8); return x;
}
static inline uint32_t __funnelshift_l(uint32_t lo, uint32_t hi, int s) {
  return (uint32_t)((((uint64_t)hi << 32 | lo) << s) >> 32);
}
static inline float __uint_as_float(uint32_t u) { float f; memcpy(&f, &u, 4); return f; }
static inline uint32_t __float_as_uint(float f) { uint32_t u; memcpy(&u, &f, 4); return u; }
static inline int __clz(int x) { return x ? __builtin_clz((unsigned)x) : 32; }
#include "rt_convert.cuh"
static long bad = 0, n = 0;
static void down(uint64_t u) {
  double x; memcpy(&x, &u, 8);
  volatile float want = (float)x;
  const float got = rt::to_f32(x), w = want;
  ++n;
  if (x != x ? got == got : memcmp(&got, &w, 4) != 0) {
    if (bad++ < 5) printf("to_f32 %016llx: %08x, want %08x\n", (unsigned long long)u, __float_as_uint(got), __float_as_uint(w));
  }
}
static void up(uint32_t u) {
  const float f = __uint_as_float(u);
  volatile double want = f;
  const double got = rt::to_f64(f), w = want;
  ++n;
  if (f != f ? got == got : bits(got) != bits(w)) {
    if (bad++ < 5) printf("to_f64 %08x: %016llx, want %016llx\n", u, (unsigned long long)bits(got), (unsigned long long)bits(w));
  }
}
int main() {
  uint64_t s = 0x9e3779b97f4a7c15ull;
  auto rnd = [&] { s ^= s << 13; s ^= s >> 7; s ^= s << 17; return s; };
  for (int i = 0; i < 2000000; ++i) { down(rnd()); up((uint32_t)rnd()); }
  for (int e = 0; e < 2048; ++e)
    for (int b = 0; b < 53; ++b)
      for (int k = 0; k < 24; ++k) {   // a leading part, a one at bit b, and the numbers next to it
        uint64_t m = k < 8 ? 0 : k < 16 ? rnd() : ~0ull;
        m = (m >> b << b | (b ? 1ull << (b - 1) : 0)) + (uint64_t)(k % 3) - 1;
        down((uint64_t)(k & 1) << 63 | (uint64_t)e << 52 | (m & 0xfffffffffffffull));
        if (e >= 860 && e <= 1160) down((uint64_t)e << 52 | (rnd() & 0xfffffffffffffull));
      }
  for (uint32_t e = 0; e < 256; ++e)
    for (uint32_t k = 0; k < 4096; ++k) up((k & 1) << 31 | e << 23 | (k < 2048 ? (uint32_t)rnd() & 0x7fffff : k < 3000 ? k - 2048 : 0x7fffff - (k - 3000)));
  printf("%ld of %ld differ\n", bad, n);
  return bad != 0;
}
"""


@pytest.mark.skipif(shutil.which("g++") is None, reason="needs a host compiler")
def test_integer_conversions_have_the_bits_of_the_hardware_ones(tmp_path):
    src = tmp_path / "convert.cpp"
    src.write_text(HOST)
    exe = str(tmp_path / "convert")
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", CSRC, str(src), "-o", exe], check=True)
    r = subprocess.run([exe], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout
