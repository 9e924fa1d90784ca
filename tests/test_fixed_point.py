"""The block fixed-point storage of the float-float solutions (hp_fixed.cuh), compiled for the host, against FP64.

Sites of 24 components whose magnitudes span up to six decades, float-float values with full low parts.  Bounds, in units
of the site's largest component: stored value 2^-51 (the remainder of a component below 2^23 units is rounded at 2^-25
units, and the largest component has at least 2^26), every bit where the component is within 1/8 of the largest; value read back
as float-float 2^-48, and where FP32 ends (sites below 2^-99) the rounding of the two parts to its smallest number, 2^-149.
"""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1302_4018_gb300", "csrc")

HARNESS = r"""
#include <cmath>
#include <cstdio>
#include <cstring>
#include <random>
#define __device__
#define __forceinline__ inline
static int __float_as_int(float f) { int i; std::memcpy(&i, &f, 4); return i; }
static float __int_as_float(int i) { float f; std::memcpy(&f, &i, 4); return f; }
static int __float2int_rn(float f) { return (int)std::nearbyintf(f); }
static float __fadd_rn(float a, float b) { return a + b; }
static float __fsub_rn(float a, float b) { return a - b; }
#include "hp_fixed.cuh"
int main() {
  std::mt19937_64 g(17);
  std::uniform_real_distribution<double> u(-1.0, 1.0), w(0.0, 1.0);
  double stored = 0.0, inexact = 0.0, read = 0.0, rem = 0.0;
  long big = 0;
  for (int site = 0; site < 200000; ++site) {
    const double scale = std::pow(10.0, 30.0 * u(g)), span = 6.0 * (site % 7) / 6.0;
    float hi[24], lo[24], m = 0.f, unit, inv;
    for (int k = 0; k < 24; ++k) {
      const double v = scale * u(g) * std::pow(10.0, -span * w(g));
      hi[k] = (float)v;
      lo[k] = (float)(v - hi[k]);
      m = std::fmax(m, std::fabs(hi[k]));
    }
    fix_unit(m, unit, inv);
    for (int k = 0; k < 24; ++k) {
      int i;
      float l, h, r;
      fix_split(hi[k], lo[k], inv, i, l);
      fix_value(i, l, unit, h, r);
      const double v = (double)hi[k] + lo[k], s = ((double)i + l) * unit;
      rem = std::fmax(rem, std::fabs((double)l));
      big = std::labs((long)i) > big ? std::labs((long)i) : big;
      stored = std::fmax(stored, std::fabs(s - v) / m);
      if (std::fabs(hi[k]) >= m / 8) inexact = std::fmax(inexact, std::fabs(s - v));
      read = std::fmax(read, std::fmax(0.0, std::fabs(((double)h + r) - s) - 0x1p-149) / m);
    }
  }
  std::printf("stored 2^%.2f  near the largest %g  read 2^%.2f  |l| %.3f  |i| %ld\n", std::log2(stored), inexact,
              std::log2(read), rem, big);
  return !(stored <= 0x1p-51 && inexact == 0.0 && read <= 0x1p-48 && rem < 5.0 && big <= 1L << 27);
}
"""


def test_stored_and_read_values_against_fp64(tmp_path):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no host compiler")
    src, exe = tmp_path / "fixed.cpp", tmp_path / "fixed"
    src.write_text(HARNESS)
    subprocess.run([cxx, "-std=c++17", "-O1", "-ffp-contract=off", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout + r.stderr
