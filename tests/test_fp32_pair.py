"""Arithmetic of float pairs (csrc/fp32_pair.cuh, compiled for the host) against
long double: quotients are the exact ones rounded to FP32 unless those lie within
2^-40 of the middle of two floats, over the whole exponent range and with the
starting reciprocal at the ends of its error bound (2^-21; products and sums lose
at most 2^-44 of their larger operand)."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(__file__), "..", "paper_2408_03452_gb300", "csrc")

SRC = r"""
#include "fp32_pair.cuh"
#include <cstdio>
#include <random>
using namespace tpfa;
typedef long double LD;
static std::mt19937_64 g(1);
static Dfl draw(int elo, int ehi) {
  const LD v = std::ldexp((LD)((g() >> 1) | (1ull << 62)), (int)(elo + (int)(g() % (unsigned)(ehi - elo + 1))) - 62);
  const float h = (float)v;
  return {h, (float)(v - (LD)h)};
}
static LD val(Dfl a) { return (LD)a.h + (LD)a.l; }
// b as close to the exact q as FP32 allows, or q within 2^-40 of a midpoint
static bool rounded(float b, LD q) {
  const float w = (float)q;
  if (b == w) return true;
  return (float)(q * (1 + 0x1p-40L)) == b || (float)(q * (1 - 0x1p-40L)) == b;
}
int main() {
  long bad = 0;
  for (int i = 0; i < 1000000; ++i) {
    const Dfl a = draw(-50, 49), b = draw(-50, 49);
    for (int d = -2; d <= 2; ++d) {
      const float y = (1.0f / b.h) * (1.0f + d * 0x1p-23f);
      bad += !rounded(df_quot_mid(a, b, y), val(a) / val(b));
    }
    // the scaled way, over all exponents; results in the normal range
    const Dfl c = draw(-149, 126), e = draw(-149, 126);
    int kc, ke;
    const Dfl cs = df_split(c, &kc), es = df_split(e, &ke);
    if (c.h >= 0x1p-126f) bad += std::ldexp(val(cs), kc) != val(c) && c.l != 0 && std::fabs(c.l) >= 0x1p-126f;
    if (!(c.h > 0) || !(e.h > 0)) continue;
    bad += !(cs.h >= 1.f && cs.h < 2.f && std::ldexp((LD)cs.h, kc) == (LD)c.h);
    const LD q = val(c) / val(e);
    const float r = df_scale(df_quot_mid(cs, es, 1.0f / es.h), kc - ke);
    if (q >= 0x1p-125L && q < 0x1p127L) bad += !rounded(r, q);
    else if (q >= 0x1p129L) bad += !std::isinf(r);
    else if (q < 0x1p-151L) bad += r != 0.f;
    // sums and products
    const Dfl s = df_add(a, {-b.h, -b.l}), p = df_mulf(a, b.h);
    const LD big = val(a) > val(b) ? val(a) : val(b);
    bad += std::fabs(val(s) - (val(a) - val(b))) > 0x1p-44L * big;
    if (a.h * b.h > 0x1p-70f && a.h * b.h < 0x1p120f)
      bad += std::fabs(val(p) - val(a) * (LD)b.h) > 0x1p-44L * val(a) * b.h;
  }
  const Dfl zero = {0.f, 0.f};
  int k;
  bad += df_split(zero, &k).h != 0.f;
  std::printf("%ld\n", bad);
}
"""


def test_pair_arithmetic(tmp_path):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no g++")
    src, exe = tmp_path / "pair.cpp", tmp_path / "pair"
    src.write_text(SRC)
    subprocess.run([cxx, "-O2", "-std=c++17", "-ffp-contract=off", "-I", CSRC, "-o", str(exe), str(src)],
                   check=True)
    assert subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.strip() == "0"
