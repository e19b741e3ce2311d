"""CPU: what is set once is set on every device that is used (csrc/stf_once.h)."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2305_05810_gb300", "csrc")
CUDA = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "include")

SOURCE = r"""
#include "stf_once.h"
static int device;      // in place of the runtime's library
extern "C" cudaError_t cudaGetDevice(int* d) { *d = device; return device < 0 ? cudaErrorNoDevice : cudaSuccess; }
int main() {
  static stf::OncePerDevice once;
  int calls[66] = {};
  auto set = [&] { ++calls[device]; return cudaSuccess; };
  for (int k = 0; k < 3; ++k)
    for (device = 0; device < 64; device += 7) if (once(set) != cudaSuccess) return 1;
  for (device = 0; device < 64; ++device) if (calls[device] != (device % 7 == 0)) return 2;
  device = 65;
  for (int k = 0; k < 2; ++k) once(set);
  if (calls[65] != 2) return 3;
  device = 1;           // a failure is tried again
  if (once([] { return cudaErrorInvalidValue; }) != cudaErrorInvalidValue) return 4;
  once(set); once(set);
  if (calls[1] != 1) return 5;
  device = -1;
  return once(set) == cudaErrorNoDevice ? 0 : 6;
}
"""


def test_every_device_is_set_once(tmp_path):
    cxx = shutil.which("g++")
    if cxx is None or not os.path.exists(os.path.join(CUDA, "cuda_runtime_api.h")):
        pytest.skip("no C++ compiler or no CUDA headers")
    src, exe = tmp_path / "once.cpp", str(tmp_path / "once")
    src.write_text(SOURCE)
    subprocess.check_call([cxx, "-std=c++17", "-I" + CSRC, "-I" + CUDA, str(src), "-o", exe])
    assert subprocess.run([exe]).returncode == 0


def test_kernel_attributes_are_set_per_device():
    """Limits of a kernel belong to a device: no plain flag keeps them from a second one."""
    for name in os.listdir(CSRC):
        with open(os.path.join(CSRC, name)) as f:
            lines = f.read().split("\n")
        for i, line in enumerate(lines):
            if "cudaFuncSetAttribute(" in line:
                assert any("OncePerDevice" in l or "once(" in l for l in lines[max(0, i - 3):i + 1]), (name, i + 1)
