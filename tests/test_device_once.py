"""Host check of the per-device cache behind the kernels' shared-memory limits
(csrc/device_once.h): a second device is configured too, a failure is not
remembered, and threads that race set once."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_1508_02766_gb300", "csrc")

PROG = r"""
#include <cstdio>
#include <thread>
#include <vector>
#include "device_once.h"
int main() {
  kde::DeviceOnce once;
  int a = 0, b = 0, calls = 0, fail = 1;
  auto set = [&] { ++calls; return 0; };
  once.run<int>(0, &a, set);
  once.run<int>(0, &a, set);
  std::printf("%d ", calls);          // 1
  once.run<int>(1, &a, set);          // the same kernel, another device
  once.run<int>(0, &b, set);          // another kernel
  once.run<int>(1, &a, set);
  std::printf("%d ", calls);          // 3
  auto bad = [&] { ++calls; return fail; };
  std::printf("%d ", once.run<int>(1, &b, bad));
  fail = 0;
  std::printf("%d ", once.run<int>(1, &b, bad));
  std::printf("%d ", once.run<int>(1, &b, bad));
  std::printf("%d ", calls);          // 5
  std::vector<std::thread> t;
  for (int i = 0; i < 8; ++i) t.emplace_back([&] { for (int d = 2; d < 6; ++d) once.run<int>(d, &a, set); });
  for (auto& x : t) x.join();
  std::printf("%d\n", calls);         // 9
  return 0;
}
"""


def test_once_per_device_and_kernel(tmp_path):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no g++")
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(PROG)
    subprocess.run([gxx, "-std=c++17", "-O2", "-pthread", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split()
    assert out == ["1", "3", "1", "0", "0", "5", "9"]


def test_every_kernel_limit_is_kept_per_device():
    """No launcher remembers a kernel's limit in a flag of its own: the limits
    are set through smem_limit.cuh, or on every call."""
    for f in os.listdir(CSRC):
        text = open(os.path.join(CSRC, f)).read()
        assert "static bool attr" not in text, f
        if f not in ("smem_limit.cuh", "bin.cu", "line1d.cu"):
            assert "cudaFuncAttributeMaxDynamicSharedMemorySize" not in text, f
