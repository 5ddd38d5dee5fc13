"""The quotient digits of the integer division (csrc/fp64_div.cuh, compiled for the
host) against the hardware's division, with the starting reciprocal at the ends of
its error bound."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(__file__), "..", "paper_2408_03452_gb300", "csrc")

SRC = r"""
#include "fp64_div.cuh"
#include <cstdio>
#include <random>
int main() {
  std::mt19937_64 g(1);
  const uint64_t one = 1ull << 52;
  auto draw = [&]() -> uint64_t {
    uint64_t r = g() & (one - 1);
    switch (g() % 5) {
      case 0: r &= ~0ull << (g() % 52); break;
      case 1: r |= (1ull << (g() % 52)) - 1; break;
      case 2: r = g() % 64; break;
      case 3: r = one - 1 - g() % 64; break;
    }
    return (r & (one - 1)) | one;
  };
  long bad = 0;
  for (int i = 0; i < 1000000; ++i) {
    const uint64_t a = draw(), b = draw();
    const double q = (double)a / (double)b;
    uint64_t want;
    memcpy(&want, &q, 8);
    want = (want & (one - 1)) | one;
    const uint32_t xb = 0x3f800000u | ((uint32_t)(b >> 29) & 0x7fffffu);
    float x;
    memcpy(&x, &xb, 4);
    for (int d = -2; d <= 2; ++d) {  // +- 2 units in the last place
      float y = 1.0f / x;
      uint32_t u;
      memcpy(&u, &y, 4);
      u += d;
      memcpy(&y, &u, 4);
      bad += tpfa::div_digits(a < b ? a << 1 : a, b, y) != want;
    }
  }
  std::printf("%ld\n", bad);
}
"""


def test_quotient_digits(tmp_path):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no g++")
    src, exe = tmp_path / "div.cpp", tmp_path / "div"
    src.write_text(SRC)
    subprocess.run([cxx, "-O2", "-std=c++17", "-I", CSRC, "-o", str(exe), str(src)], check=True)
    assert subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.strip() == "0"
