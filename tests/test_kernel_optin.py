"""Kernel attributes (the shared memory above 48 KB) belong to a device, so the
record of what was set belongs to the library context (csrc/optin.h), never to
the process: compiled for the host with a stand-in for the CUDA call."""
import os
import re
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2305_07181_gb300", "csrc")

MAIN = r"""
#include "optin.h"
#include <cstdio>
#include <thread>
#include <vector>
int main() {
  static char kernels[64];
  int device = 0, sets[2] = {0, 0}, refuse = 0;
  auto launch = [&](esplit::OptIn& o, int k) {
    return o.once(&kernels[k], [&]() -> int { if (refuse) return -7; ++sets[device]; return 0; });
  };
  esplit::OptIn a, b;  // contexts on device 0 and device 1
  for (int i = 0; i < 3; ++i) launch(a, 0);
  device = 1;
  for (int i = 0; i < 3; ++i) launch(b, 0);
  std::printf("%d %d\n", sets[0], sets[1]);
  refuse = 1;  // a refusal reaches the caller and is not remembered
  const int first = launch(b, 1), second = launch(b, 1);
  refuse = 0;
  const int third = launch(b, 1);
  std::printf("%d %d %d %d\n", first, second, third, sets[1]);
  esplit::OptIn c;  // more kernels than it records: each of them is set at least once
  sets[1] = 0;
  for (int k = 0; k < 64; ++k) launch(c, k);
  std::printf("%d\n", sets[1]);
  esplit::OptIn d;  // several threads on one context: set once
  int n = 0;
  std::vector<std::thread> t;
  for (int k = 0; k < 8; ++k) t.emplace_back([&]() { for (int i = 0; i < 1000; ++i) d.once(kernels, [&]() -> int { ++n; return 0; }); });
  for (auto& x : t) x.join();
  std::printf("%d\n", n);
}
"""


def test_set_once_per_context(tmp_path):
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("no g++")
    src = tmp_path / "m.cpp"
    src.write_text(MAIN)
    exe = str(tmp_path / "m")
    subprocess.run([cxx, "-O1", "-std=c++17", "-pthread", "-I", CSRC, str(src), "-o", exe], check=True)
    out = subprocess.run([exe], capture_output=True, text=True, check=True).stdout.split("\n")
    assert out[:4] == ["1 1", "-7 -7 0 2", "64", "1"]


def test_no_kernel_remembers_its_attributes_by_itself():
    for name in sorted(os.listdir(CSRC)):
        if not name.endswith((".cu", ".cuh", ".h")) or name == "internal.h":
            continue
        with open(os.path.join(CSRC, name)) as f:
            text = f.read()
        assert "cudaFuncSetAttribute(" not in text, name     # internal.h: opt_in_smem, the one place
        assert not re.search(r"static\s+(bool|int|size_t)\s+\w*(attr|carve)\w*\s*=", text), name
