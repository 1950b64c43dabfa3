"""once_per_device.h: what belongs to a device is set on each device that is used, once if it
succeeds and again if it failed (compiled here for the host, with made-up devices; kernels'
shared-memory limits are set through it)."""
import os
import re
import subprocess

from tests._util import ROOT

CSRC = os.path.join(ROOT, "paper_2504_12217_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include <vector>
#include "once_per_device.h"
int main() {
  zkvc::OncePerDevice once;
  std::vector<int> calls(70, 0);
  auto ask = [&](int dev, int status) { return once(dev, [&] { calls[dev]++; return status; }); };
  int bad = 0;
  bad += ask(0, 0) != 0 || ask(0, 0) != 0 || calls[0] != 1;    // once
  bad += ask(1, 0) != 0 || calls[1] != 1;                      // another device: its own
  bad += ask(7, -3) != -3 || ask(7, -3) != -3 || calls[7] != 2;  // a failure is reported and not kept
  bad += ask(7, 0) != 0 || ask(7, 0) != 0 || calls[7] != 3;
  bad += ask(63, 0) != 0 || ask(63, 0) != 0 || calls[63] != 1;
  bad += ask(69, 0) != 0 || ask(69, 0) != 0 || calls[69] != 2;  // past what is remembered: every time
  bad += ask(0, -1) != 0 || ask(1, -1) != 0 || calls[0] != 1 || calls[1] != 1;
  std::printf("%d\n", bad);
  return bad;
}
"""


def test_once_per_device(tmp_path):
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    assert subprocess.run([str(exe)], capture_output=True, text=True).stdout == "0\n"


def test_shared_memory_limits_go_through_it():
    """No unit sets a kernel's attribute but through smem_limits, which reports its errors."""
    for name in sorted(os.listdir(CSRC)):
        text = open(os.path.join(CSRC, name)).read()
        if name != "internal.h":
            assert "cudaFuncSetAttribute" not in text, name
        else:
            assert re.search(r"ZK_CUDA\(cudaFuncSetAttribute\(", text)
