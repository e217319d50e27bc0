"""Sums of an offset and a displacement in two FP32 parts (csrc/sph_disp.cuh) on the
CPU: equal to the FP64 form, also next to a tie."""
import os
import shutil
import subprocess

import pytest

from paper_2104_00537_gb300 import build

SRC = r"""
#include <cstdint>
#include <cstdio>
#include <random>
#include "sph_disp.cuh"
using namespace sph;
static long bad = 0;
static void check(float off, const Disp &d, double disp) {
  const float want = (float)((double)off + disp), got = add_disp(off, d);
  if (got != want && bad++ < 5) std::printf("%a %a + %a: %a, not %a\n", off, d.hi, d.lo, got, want);
}
int main() {
  std::mt19937_64 g(5);
  std::uniform_real_distribution<double> U(0, 1);
  // half a unit of the offset and a little more or less, either sign
  for (int k = 0; k < 20000; k++) {
    const float off = (float)(0.01 + 0.1 * U(g));
    const float half = 0.5f * (nextafterf(off, 1.f) - off);
    for (int q = 0; q < 4; q++) {
      const float hi = (q & 1 ? -1.f : 1.f) * half, lo = (q & 2 ? -1.f : 1.f) * half * 0x1p-26f;
      check(off, Disp{hi, lo}, (double)hi + (double)lo);
    }
  }
  // a step's products: dt in two parts times a velocity (and dt^2 / 2 times an
  // acceleration, the Verlet scheme's), offsets in a cell and near its lower face
  for (int k = 0; k < 3000000; k++) {
    const double cs = 0.008 * std::pow(18.0, U(g)), dt = 1e-6 * std::pow(1e3, U(g));
    float off = (float)(U(g) * cs), v = (float)((2 * U(g) - 1) * 5), a = (float)((2 * U(g) - 1) * 500);
    if (k % 4 == 0) off *= (float)std::pow(2.0, -20 * U(g));
    const double dt2 = 0.5 * dt * dt;
    const float c[2] = {(float)dt, (float)(dt - (double)(float)dt)};
    const float c2[2] = {(float)dt2, (float)(dt2 - (double)(float)dt2)};
    check(off, disp_scaled(c, v), dt * (double)v);
    check(off, disp_sum(disp_scaled(c, v), disp_scaled(c2, a)),
          std::fma(dt2, (double)a, dt * (double)v));
    check(off, disp_of(dt * (double)v), dt * (double)v);
  }
  std::printf("%ld\n", bad);
  return bad != 0;
}
"""


@pytest.mark.skipif(shutil.which("g++") is None, reason="needs g++")
def test_sum_equals_fp64(tmp_path):
    src, exe = tmp_path / "d.cpp", tmp_path / "d"
    src.write_text(SRC)
    cuda = os.path.dirname(os.path.dirname(os.path.realpath(build.nvcc())))
    subprocess.run(["g++", "-std=c++17", "-O2", "-ffp-contract=off", "-I", build.CSRC, "-I",
                    os.path.join(cuda, "include"), str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
