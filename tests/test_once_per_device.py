"""What is set up once per device is set up on every device (CPU only, fake device numbers)."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2507_18969_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include <thread>
#include <vector>
#include "once.cuh"
#define CHECK(x) if (!(x)) { std::printf("line %d: %s\n", __LINE__, #x); return 1; }
int main() {
  static edpc::OncePerDevice once;
  int calls[2] = {}, fail = 1;
  auto set = [&](int dev) { return once.run(dev, [&] { ++calls[dev]; return dev == 1 && fail-- > 0 ? 7 : 0; }); };
  CHECK(set(0) == 0 && set(0) == 0 && calls[0] == 1);
  CHECK(set(1) == 7 && calls[1] == 1);                  // a second device is set up too, and a failure is told
  CHECK(set(1) == 0 && set(1) == 0 && calls[1] == 2);   // ... and tried again, until it succeeds
  CHECK(set(0) == 0 && calls[0] == 1);
  int beyond = 0;
  for (int dev : {-1, edpc::OncePerDevice::kDevices}) CHECK(once.run(dev, [&] { ++beyond; return 0; }) == 0);
  CHECK(beyond == 2);
  static edpc::OncePerDevice shared;
  std::atomic<int> n{0};
  std::vector<std::thread> th;
  for (int t = 0; t < 8; ++t)
    th.emplace_back([&] { for (int dev = 0; dev < 64; ++dev) shared.run(dev, [&] { ++n; return 0; }); });
  for (auto& t : th) t.join();
  CHECK(n == 64);
  return 0;
}
"""


def test_each_device_is_set_up_once(tmp_path):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no g++")
    src, exe = tmp_path / "once.cpp", tmp_path / "once"
    src.write_text(PROGRAM)
    subprocess.run([cxx, "-std=c++17", "-O1", "-pthread", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout


def test_no_attribute_is_set_once_per_process():
    """Kernel attributes hold for the current device only."""
    for name in sorted(os.listdir(CSRC)):
        if name.endswith((".cu", ".cuh")):
            src = open(os.path.join(CSRC, name)).read()
            for part in src.split("std::call_once")[1:]:
                body = part[:part.index("});")]
                assert "cudaFuncSetAttribute" not in body and "cudaDeviceGetAttribute" not in body, name
