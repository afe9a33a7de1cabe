"""The conversions on the integer units give the bits of the plain casts.

widen() and narrow() (csrc/convert_bits.cuh) replace (double)f and (float)d where a pass over whole
vectors would be bound by the conversion instructions. The header is plain C++ and is compiled here
for the host: every exponent and sign with mantissas at the rounding boundaries, every special value
and random bit patterns have to agree bit for bit with the casts (a NaN has to stay a NaN).
"""

import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SRC = r"""
#include "convert_bits.cuh"
#include <cstdio>
#include <random>
static uint64_t b64(double d) { uint64_t u; std::memcpy(&u, &d, 8); return u; }
static uint32_t b32(float f) { uint32_t u; std::memcpy(&u, &f, 4); return u; }
static double d64(uint64_t u) { double d; std::memcpy(&d, &u, 8); return d; }
static float f32(uint32_t u) { float f; std::memcpy(&f, &u, 4); return f; }
static long bad = 0;
static void w(float f) {
  const double a = wdf::widen(f), b = (double)f;
  if (b != b ? a == a : b64(a) != b64(b)) ++bad;
}
static void n(double d) {
  const float a = wdf::narrow(d), b = (float)d;
  if (b != b ? a == a : b32(a) != b32(b)) ++bad;
}
int main() {
  std::mt19937_64 g(7);
  const uint64_t mant[] = {0, 1, 0xFFFFFFF, 0x10000000, 0x10000001, 0x1FFFFFFF, 0x20000000, 0x2FFFFFFF, 0x30000000, 0x30000001, 0x3FFFFFFF,
                           0xFFFFFEFFFFFFFull, 0xFFFFFF0000000ull, 0xFFFFFFFFFFFFFull, 0x8000000000000ull};
  for (uint64_t e = 0; e < 2048; ++e)
    for (uint64_t s = 0; s < 2; ++s) {
      for (uint64_t m : mant) n(d64(s << 63 | e << 52 | m));
      for (int k = 0; k < 500; ++k) n(d64(s << 63 | e << 52 | (g() >> 12)));
    }
  for (uint32_t e = 0; e < 256; ++e)
    for (uint32_t s = 0; s < 2; ++s) {
      for (uint32_t m : {0u, 1u, 2u, 0x400000u, 0x7FFFFFu}) w(f32(s << 31 | e << 23 | m));
      for (int k = 0; k < 2000; ++k) w(f32(s << 31 | e << 23 | (uint32_t)(g() >> 41)));
    }
  std::printf("%ld\n", bad);
  return bad != 0;
}
"""


@pytest.mark.skipif(shutil.which("g++") is None, reason="needs g++")
def test_integer_conversions_have_the_bits_of_the_casts(tmp_path):
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(SRC)
    inc = os.path.join(ROOT, "paper_2607_14025_gb300", "csrc")
    subprocess.run(["g++", "-O2", "-std=c++17", "-Wall", "-Werror", "-I", inc, str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0 and r.stdout.strip() == "0", r.stdout
