"""The check kernels' float/double conversions and comparison in integer operations
(csrc/conv_bits.h) equal the hardware's bit for bit: every exponent of a float, every
exponent around a float's range of a double, with mantissas at the rounding's edges."""
import os
import shutil
import subprocess

import pytest

from paper_2307_03466_gb300 import build as B

SOURCE = r"""
#include <cmath>
#include <cstdio>
#include <cstring>
#include <initializer_list>
#include "conv_bits.h"
template <typename A, typename C> static A as(C c) { A a; std::memcpy(&a, &c, sizeof a); return a; }
int main() {
  long bad = 0;
  const uint32_t fm[] = {0, 1, 2, 3, 0x3fffff, 0x400000, 0x400001, 0x555555, 0x7ffffe, 0x7fffff};
  for (uint32_t e = 0; e < 256; ++e)
    for (uint32_t m : fm)
      for (uint32_t s = 0; s < 2; ++s) {
        const float f = as<float>(s << 31 | e << 23 | m);
        const bool small = std::fabs(f) < 0x1p-100f;
        const double d = as<double>(scylla::f64_bits(as<uint32_t>(small ? f * 0x1p100f : f), small));
        bad += std::isnan(f) ? !std::isnan(d) : as<uint64_t>(d) != as<uint64_t>(double(f));
      }
  for (uint64_t e = 0; e < 2048; ++e)
    for (uint64_t top : {0ull, 1ull, 2ull, 0x7ffffeull, 0x7fffffull, 0x2aaaaaull})
      for (uint64_t low : {0ull, 1ull, 0xfffffffull, 0x10000000ull, 0x10000001ull, 0x1fffffffull})
        for (uint64_t s = 0; s < 2; ++s) {
          const double d = as<double>(s << 63 | e << 52 | top << 29 | low);
          const float f = as<float>(scylla::f32_bits(as<uint64_t>(d)));
          bad += std::isnan(d) ? !std::isnan(f) : as<uint32_t>(f) != as<uint32_t>(float(d));
        }
  const double v[] = {-INFINITY, -1e300, -1.5, -1.0, -5e-324, -0.0, 0.0, 5e-324, 1.0, 1.5, 1e300, INFINITY};
  for (int i = 0; i < 12; ++i)  // in ascending order, -0 below +0
    for (int j = 0; j < 12; ++j) bad += scylla::f64_less_bits(as<int64_t>(v[i]), as<int64_t>(v[j])) != (i < j);
  std::printf("%ld\n", bad);
}
"""


def test_conversions_equal_the_hardware(tmp_path):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("needs g++")
    src, exe = tmp_path / "h.cpp", tmp_path / "h"
    src.write_text(SOURCE)
    subprocess.run([cxx, "-O2", "-std=c++17", "-I", B.CSRC, str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0 and r.stdout.strip() == "0", r.stdout + r.stderr
