"""CPU check of the integer conversions between FP64 and FP32 that the FP32
storage's FP64 wide terms use: the functions of f32_convert.cuh, compiled for the
host, against plain casts, bit for bit (subnormals as zero, a NaN of FP64 arithmetic as NaN)."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1703_00185_gb300", "csrc")

PROGRAM = r"""
#define __host__
#define __device__
#define __forceinline__ inline
#include <cmath>
#include <cstdio>
#include <cstring>
#include <initializer_list>
#include "f32_convert.cuh"
using namespace d2q37;
static long bad = 0, seen = 0;
static void narrow(uint64_t u) {
  double v;
  std::memcpy(&v, &u, 8);
  const uint32_t got = f32_bits((uint32_t)(u >> 32), (uint32_t)u);
  ++seen;
  if (std::isnan(v)) {  // made by arithmetic: a payload in the high word
    if ((u >> 32 & 0x7FFFFFFF) > 0x7FF00000) bad += !((got & 0x7F800000u) == 0x7F800000u && (got & 0x7FFFFFu));
    return;
  }
  const float c = std::fabs(v) < 0x1p-126 ? std::copysign(0.0f, (float)v) : (float)v;
  uint32_t want;
  std::memcpy(&want, &c, 4);
  if (got != want && bad++ < 5) std::printf("narrow %016llx %08x %08x\n", (unsigned long long)u, got, want);
}
static void widen(uint32_t b) {
  float v;
  std::memcpy(&v, &b, 4);
  const uint64_t got = (uint64_t)f64_high(b) << 32 | f64_low(b);
  ++seen;
  if (std::isnan(v)) {
    bad += !((got << 1 >> 53) == 0x7FFu && (got & 0xFFFFFFFFFFFFFull));
    return;
  }
  const double c = (b & 0x7F800000u) ? (double)v : std::copysign(0.0, (double)v);
  uint64_t want;
  std::memcpy(&want, &c, 8);
  if (got != want && bad++ < 5) std::printf("widen %08x\n", b);
}
int main() {
  uint64_t s = 1;
  for (uint32_t e = 0; e < 2048; ++e)  // every exponent, ties and their neighbours, carries, both signs
    for (uint64_t top : {0ull, 1ull, 2ull, 3ull, 0x7FFFFEull, 0x7FFFFFull})
      for (uint64_t low : {0ull, 1ull, 0xFFFFFFFull, 0x10000000ull, 0x10000001ull, 0x1FFFFFFFull})
        for (uint64_t sign : {0ull, 1ull}) narrow(sign << 63 | (uint64_t)e << 52 | top << 29 | low);
  for (long k = 0; k < 3000000; ++k) {
    s = s * 6364136223846793005ull + 1442695040888963407ull;
    narrow(s);
    narrow((s & 0x800FFFFFFFFFFFFFull) | (uint64_t)(890 + k % 270) << 52);  // around the range of a float
    narrow((s & 0xFFFFFFFFF0000000ull));                                   // ties
  }
  for (uint64_t b = 0; b < (1ull << 32); b += 251) widen((uint32_t)b);
  for (uint32_t b : {0u, 1u, 0x7FFFFFu, 0x800000u, 0x7F7FFFFFu, 0x7F800000u, 0x7F800001u, 0x7F800007u, 0x7FC00000u}) widen(b), widen(b | 0x80000000u);
  std::printf("%ld of %ld differ\n", bad, seen);
  return bad != 0;
}
"""


@pytest.mark.skipif(shutil.which("g++") is None, reason="needs g++")
def test_integer_conversions_are_the_casts(tmp_path):
    src = tmp_path / "t.cpp"
    src.write_text(PROGRAM)
    exe = tmp_path / "t"
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
