"""The composite's colour sums for every group size, compiled for the host with bounds checks on its arrays
(no GPU needed): a group's channels are not a multiple of the 16-byte words that its colours are read in."""
import os
import shutil
import subprocess

import pytest

from paper_2408_03538_gb300 import build as B

SOURCE = r"""
#include <cmath>
#include <cstdio>
#include "blend.cuh"
using namespace prtgs;
template <int KG>
static int check() {
  alignas(16) float row[color_floats(KG)];
  float acc[3 * KG];
  for (int e = 0; e < color_floats(KG); ++e) row[e] = e < 3 * KG ? 1.0f + e : NAN;  // the padding reaches no sum
  for (int e = 0; e < 3 * KG; ++e) acc[e] = 100.0f * e;
  blend_row<KG>(acc, row, 0.5f);
  for (int e = 0; e < 3 * KG; ++e)
    if (acc[e] != 100.0f * e + 0.5f * (1.0f + e)) return 1;
  return 0;
}
int main() {
  const int bad = check<1>() + check<2>() + check<4>() + check<8>() + check<16>();
  std::puts(bad ? "wrong sums" : "ok");
  return bad;
}
"""


def test_blend_row_stays_inside_its_sums(tmp_path):
    if shutil.which("g++") is None:
        pytest.skip("no host compiler")
    src, exe = tmp_path / "blend.cu", tmp_path / "blend"
    src.write_text(SOURCE)
    flags = ["-O0", "-std=c++17", "-I", B.CSRC, "-Xcompiler", "-fsanitize=bounds,-fno-sanitize-recover=all"]
    r = subprocess.run([B.nvcc(), *B.ARCH, *flags, str(src), "-o", str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    out = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60, cwd=os.fspath(tmp_path))
    assert out.returncode == 0 and out.stdout.strip() == "ok", out.stdout + out.stderr
