"""CPU: which arrays count as the current device's own memory (csrc/stf_memory.h)."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2305_05810_gb300", "csrc")
CUDA = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "include")

SOURCE = r"""
#include <cstdio>
// the attributes as the runtime would give them: in place of its library
#include "stf_memory.h"
static cudaPointerAttributes at;
static cudaError_t result = cudaSuccess;
extern "C" {
cudaError_t cudaPointerGetAttributes(cudaPointerAttributes* a, const void*) { *a = at; return result; }
cudaError_t cudaGetDevice(int* d) { *d = 1; return cudaSuccess; }
cudaError_t cudaGetLastError() { return result; }
}
int main() {
  int x = 0;
  const cudaMemoryType types[] = {cudaMemoryTypeUnregistered, cudaMemoryTypeHost, cudaMemoryTypeDevice, cudaMemoryTypeManaged};
  for (auto t : types)
    for (int d = 0; d < 3; ++d) {
      at.type = t;
      at.device = d;
      if (stf::local_memory(&x) != (t == cudaMemoryTypeDevice && d == 1)) return 1;
    }
  at.type = cudaMemoryTypeDevice;
  at.device = 1;
  if (stf::local_memory(nullptr)) return 2;
  result = cudaErrorInvalidValue;
  return stf::local_memory(&x) ? 3 : 0;
}
"""


def test_only_the_current_devices_memory_is_local(tmp_path):
    cxx = shutil.which("g++")
    if cxx is None or not os.path.exists(os.path.join(CUDA, "cuda_runtime_api.h")):
        pytest.skip("no C++ compiler or no CUDA headers")
    src, exe = tmp_path / "memory.cpp", str(tmp_path / "memory")
    src.write_text(SOURCE)
    subprocess.check_call([cxx, "-std=c++17", "-I" + CSRC, "-I" + CUDA, str(src), "-o", exe])
    assert subprocess.run([exe]).returncode == 0
