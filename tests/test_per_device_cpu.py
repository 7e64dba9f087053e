"""The per-device set-up of the launchers (csrc/per_device.h), compiled for the
host: a second device is set up on its own, a failure is not kept, and threads
that arrive together set a device up once."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2609_37924_gb300", "csrc")

MAIN = r"""
#include <cstdio>
#include <thread>
#include <vector>
#include "per_device.h"
#define CHECK(x) do { if (!(x)) { std::printf("line %d: %s\n", __LINE__, #x); return 1; } } while (0)
int main() {
  tadm::PerDevice p;
  int n = 0;
  CHECK(p.get(0, [&] { ++n; return 152; }) == 152 && n == 1);
  CHECK(p.get(0, [&] { ++n; return 7; }) == 152 && n == 1);
  CHECK(p.get(1, [&] { ++n; return 148; }) == 148 && n == 2);      // another device: its own set-up and value
  CHECK(p.get(0, [&] { ++n; return 7; }) == 152 && n == 2);
  CHECK(p.get(2, [&] { ++n; return -3; }) == -3 && n == 3);        // a failure is reported and tried again
  CHECK(p.get(2, [&] { ++n; return 132; }) == 132 && n == 4);
  const int past = tadm::PerDevice::kMax;
  CHECK(p.get(past, [&] { ++n; return 5; }) == 5 && p.get(past, [&] { ++n; return 6; }) == 6 && n == 6);
  CHECK(p.get(-1, [&] { ++n; return 9; }) == 9 && n == 7);
  tadm::PerDevice q;
  std::atomic<int> calls{0}, sum{0};
  std::vector<std::thread> ts;
  for (int t = 0; t < 8; ++t)
    ts.emplace_back([&] { for (int d = 0; d < 4; ++d) sum += q.get(d, [&] { ++calls; return d + 1; }); });
  for (auto& t : ts) t.join();
  CHECK(calls == 4 && sum == 8 * (1 + 2 + 3 + 4));
  return 0;
}
"""


def test_set_up_per_device(tmp_path):
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("no g++")
    src = tmp_path / "main.cpp"
    src.write_text(MAIN)
    exe = str(tmp_path / "main")
    subprocess.run([cxx, "-std=c++17", "-O1", "-pthread", "-I", CSRC, str(src), "-o", exe], check=True)
    r = subprocess.run([exe], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout


def test_opt_in_shared_memory_of_the_fp32_kernels_is_per_device():
    """The fp32 GEMM and attention kernels run on whichever device is current, so no process-wide flag guards their
    shared-memory attribute: each such call sits in a per-device set-up."""
    with open(os.path.join(CSRC, "gemm_simt.cu")) as f:
        gemm = f.read()
    with open(os.path.join(CSRC, "attention.cu")) as f:
        attn = f.read()
    attn = attn[attn.index("cudaError_t launch_f32("):]
    attn = attn[:attn.index("\n}\n")]
    for src in (gemm, attn):
        assert "cudaFuncSetAttribute" in src and "PerDevice" in src
        assert "static bool" not in src and "static int " not in src
