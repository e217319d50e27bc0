"""The list walk's wrapping coordinates on the CPU (csrc/sph_internal.cuh), built
with g++ and a trap on every signed overflow."""
import os
import shutil
import subprocess

import pytest

from paper_2104_00537_gb300 import build

SRC = r"""
#include <cstdint>
#include <cstdio>
#include "sph_internal.cuh"
using namespace sph;
int main(int argc, char **) {
  // pairs at every eighth of a cell over two periods of eight cells, up to four
  // cells apart: the difference is that of the unwrapped positions
  for (int64_t x = 0; x < 128; x++)
    for (int64_t d = -31; d <= 31; d++) {
      const int a = (int)(uint32_t)(x * 67108864), b = (int)(uint32_t)((x - d) * 67108864);
      const int r = argc > 1 ? a - b : walk_delta(a, b);
      if (r != d * 67108864) {
        std::printf("%lld %lld %d\n", (long long)x, (long long)d, r);
        return 1;
      }
    }
  return 0;
}
"""


@pytest.mark.skipif(shutil.which("g++") is None, reason="needs g++")
def test_walk_delta_wraps_without_signed_overflow(tmp_path):
    src, exe = tmp_path / "w.cpp", tmp_path / "w"
    src.write_text(SRC)
    cuda = os.path.dirname(os.path.dirname(os.path.realpath(build.nvcc())))
    subprocess.run(["g++", "-std=c++17", "-O1", "-fsanitize=signed-integer-overflow",
                    "-fsanitize-undefined-trap-on-error", "-I", build.CSRC, "-I", build.INCLUDE,
                    "-I", os.path.join(cuda, "include"), str(src), "-o", str(exe)], check=True)
    assert subprocess.run([str(exe)]).returncode == 0
    # a plain subtraction of the same coordinates overflows
    assert subprocess.run([str(exe), "plain"]).returncode < 0
