"""FP32 -> FP64 and back on the integer pipe (mg_common.cuh), the bit functions compiled for the host:
the casts' bits over random values of every exponent, signed zeros, the smallest and largest subnormals,
2^-126, the largest float and infinities; a NaN stays one."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include <cmath>
#include <cstdio>
#include <cstring>
#include "mg_common.cuh"
static float f32(unsigned u) { float f; memcpy(&f, &u, 4); return f; }
static unsigned bits(float f) { unsigned u; memcpy(&u, &f, 4); return u; }
static unsigned long long bits(double d) { unsigned long long u; memcpy(&u, &d, 8); return u; }
static int wide(unsigned u) {  // as mg::widen splits its argument
  const bool tiny = (u & 0x7f800000u) == 0;
  const unsigned w = bits(tiny ? f32(u) * 0x1p64f : f32(u));
  const mg::Bits64 b = mg::widen_bits(w & 0x7fffffffu, w & 0x80000000u, tiny);
  const unsigned long long got = ((unsigned long long)b.hi << 32) | b.lo;
  if (std::isnan(f32(u))) { double d; memcpy(&d, &got, 8); return !std::isnan(d); }
  return got != bits((double)f32(u));
}
static int slim(unsigned long long u) {
  double d; memcpy(&d, &u, 8);
  const float got = f32(mg::narrow_bits((unsigned)(u >> 32), (unsigned)u));
  return std::isnan(d) ? !std::isnan(got) : bits(got) != bits((float)d);
}
int main() {
  const unsigned edge[] = {0u, 1u, 2u, 0x7fffffu, 0x800000u, 0x800001u, 0x3f800000u, 0x7f7fffffu, 0x7f800000u, 0x7fc00000u, 0x7f800001u};
  long bad = 0;
  for (unsigned e : edge) bad += wide(e) + wide(e | 0x80000000u);
  unsigned long long s = 88172645463325252ull;
  for (int k = 0; k < 20000000; ++k) {
    s ^= s << 13; s ^= s >> 7; s ^= s << 17;
    bad += wide((unsigned)s) + wide((unsigned)(s >> 32) & 0x807fffffu) + slim(s);
    bad += slim((s & 0x800fffffffffffffull) | ((850ull + (s >> 40) % 320) << 52));
  }
  printf("%ld\n", bad);
  return 0;
}
"""


def test_conversions_by_bits(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("no nvcc")
    src, exe = tmp_path / "conv.cu", tmp_path / "conv"
    src.write_text(PROGRAM)
    inc = [f for d in ("paper_2602_01888_gb300/csrc", "include") for f in ("-I", os.path.join(ROOT, d))]
    subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-O2", "-std=c++17", *inc, str(src), "-o", str(exe)], check=True)
    assert int(subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout) == 0
