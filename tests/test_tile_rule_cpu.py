"""The tile rules of the GEMM dispatch (csrc/tile_rule.h), compiled for the
host: rounds are counted over the clusters that the launch will have."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2609_37924_gb300", "csrc")

MAIN = r"""
#include <cstdio>
#include "tile_rule.h"
using tadm::glu_tiles_192;
#define CHECK(x) do { if (!(x)) { std::printf("line %d: %s\n", __LINE__, #x); return 1; } } while (0)
int main() {
  CHECK(glu_tiles_192(168, 76, 224, 76));     // 3 rounds of 256 against 3 of 192
  CHECK(!glu_tiles_192(168, 76, 224, 74));    // fewer resident clusters of the narrow kernel: 4 rounds of 192
  CHECK(!glu_tiles_192(168, 84, 224, 76));    // 2 full rounds of 256
  CHECK(glu_tiles_192(168, 70, 224, 75));
  CHECK(!glu_tiles_192(76, 76, 102, 76));     // one full round of 256
  CHECK(glu_tiles_192(77, 76, 103, 76));
  CHECK(!glu_tiles_192(77, 0, 103, 76) && !glu_tiles_192(77, 76, 103, 0));
  return 0;
}
"""


def test_glu_tile_width(tmp_path):
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("no g++")
    src = tmp_path / "main.cpp"
    src.write_text(MAIN)
    exe = str(tmp_path / "main")
    subprocess.run([cxx, "-std=c++17", "-I", CSRC, str(src), "-o", exe], check=True)
    r = subprocess.run([exe], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout
