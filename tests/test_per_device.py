"""The opt-in to large dynamic shared memory is made on every device and by every kernel
that needs it (csrc/per_device.cuh, compiled here against stand-ins of the CUDA
calls)."""
import glob
import os
import re
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2404_09452_gb300", "csrc")
CUDA = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "include")

PROGRAM = r"""
#include <cstdio>
#include <thread>
#include <vector>
#include "per_device.cuh"
thread_local int current = 0;
int calls[4], failing = -1;
extern "C" cudaError_t cudaGetDevice(int *d) { *d = current; return cudaSuccess; }
extern "C" const char *cudaGetErrorString(cudaError_t) { return "failed"; }
extern "C" cudaError_t cudaFuncSetAttribute(const void *, cudaFuncAttribute, int) {
  ++calls[current];
  return current == failing ? cudaErrorInvalidValue : cudaSuccess;
}
void kernel() {}
int main() {
  dfjk::OncePerDevice once;
  const auto use = [&](int dev) {
    current = dev;
    try {
      dfjk::allow_smem(once, &kernel, 1 << 16);
      return 0;
    } catch (const dfjk::Error &) {
      return 1;
    }
  };
  int threw = 0;
  for (int dev : {0, 0, 2, 0, 2}) threw += use(dev);
  failing = 1;
  threw += use(1);
  failing = -1;
  threw += use(1);
  std::vector<std::thread> t;
  for (int k = 0; k < 8; ++k) t.emplace_back([&] { use(3); });
  for (auto &x : t) x.join();
  std::printf("%d %d %d %d %d\n", calls[0], calls[1], calls[2], calls[3], threw);
}
"""


@pytest.mark.skipif(not os.path.exists(os.path.join(CUDA, "cuda_runtime.h")), reason="needs the CUDA headers")
def test_once_on_every_device(tmp_path):
    (tmp_path / "t.cpp").write_text(PROGRAM)
    exe = str(tmp_path / "t")
    subprocess.run(["g++", "-std=c++17", "-pthread", "-I", CSRC, "-I", CUDA, "-o", exe, str(tmp_path / "t.cpp")], check=True)
    out = subprocess.run([exe], check=True, capture_output=True, text=True).stdout.split()
    assert out == ["1", "2", "1", "1", "1"]  # a failed call is made again


def test_every_opt_in_is_per_device():
    for path in glob.glob(os.path.join(CSRC, "*.cu*")):
        text = open(path).read()
        if os.path.basename(path) != "per_device.cuh":
            assert "cudaFuncSetAttribute(" not in text, path
        for name in re.findall(r"allow_smem\((\w+),", text):
            assert re.search(r"static OncePerDevice " + name + r"\b|OncePerDevice &" + name, text), path
