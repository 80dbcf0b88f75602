"""Host side of the choice between kernels and copies for a caller's array (no GPU):
another device's memory goes through copies, as pageable host memory does.  Compiled
with the host C++ compiler against csrc/kernel_address.h."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2411_09605_gb300", "csrc")
CUDA_INC = "/usr/local/cuda/include"

PROGRAM = r"""
#include <cstdio>
#include "kernel_address.h"
int main() {
  int there = 0;
  const cudaMemoryType types[] = {cudaMemoryTypeUnregistered, cudaMemoryTypeHost,
                                  cudaMemoryTypeDevice, cudaMemoryTypeManaged};
  for (cudaMemoryType t : types)
    for (int owner = 0; owner < 2; owner++) {
      cudaPointerAttributes a{};
      a.type = t;
      a.device = owner;
      a.devicePointer = t == cudaMemoryTypeUnregistered ? nullptr : &there;
      std::printf("%d", pic::kernel_address(a, 1) == &there);
    }
}
"""


def test_only_memory_that_kernels_reach(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None or not os.path.isdir(CUDA_INC):
        pytest.skip("needs a host C++ compiler and the CUDA headers")
    src, exe = tmp_path / "address.cpp", tmp_path / "address"
    src.write_text(PROGRAM)
    r = subprocess.run([cxx, "-std=c++17", "-I", CSRC, "-I", CUDA_INC, str(src), "-o", str(exe)],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    out = subprocess.run([str(exe)], capture_output=True, text=True, check=True).stdout
    assert out == "00" "11" "01" "11"   # pageable, pinned, device 0 and 1, managed
