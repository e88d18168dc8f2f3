"""The shared memory limit of a kernel is raised on every device that launches it
(the CUDA calls faked on the host: several devices in one process)."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1908_06742_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include <initializer_list>
#include "ddflb_smem.h"
static int device = 0, calls[128], fail = 0;
extern "C" cudaError_t cudaGetDevice(int* d) { *d = device; return cudaSuccess; }
extern "C" cudaError_t cudaFuncSetAttribute(const void*, cudaFuncAttribute a, int bytes) {
  if (a != cudaFuncAttributeMaxDynamicSharedMemorySize || bytes != 100000) return cudaErrorUnknown;
  ++calls[device];
  return fail ? cudaErrorInvalidValue : cudaSuccess;
}
int main() {
  ddflb::SharedLimit limit;
  int bad = 0;
  auto raise_on = [&](int d) { device = d; return limit.raise(&limit, 100000); };
  fail = 1;  // a refusal is reported, and tried again at the next launch
  if (raise_on(0) != cudaErrorInvalidValue || calls[0] != 1) bad |= 1;
  fail = 0;
  for (int round = 0; round < 3; ++round)
    for (int d : {0, 1, 7, 63, 70})
      if (raise_on(d) != cudaSuccess) bad |= 2;
  if (calls[0] != 2 || calls[1] != 1 || calls[7] != 1 || calls[63] != 1) bad |= 4;
  if (calls[70] != 3) bad |= 8;
  std::printf("%d\n", bad);
  return bad;
}
"""


def test_raised_once_per_device(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    include = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc))), "include")
    if not os.path.exists(os.path.join(include, "cuda_runtime_api.h")):
        pytest.skip("CUDA headers not found")
    src, exe = tmp_path / "limit.cpp", tmp_path / "limit"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-I", include, "-I", CSRC, str(src), "-o", str(exe)],
                   check=True)
    assert subprocess.run([str(exe)]).returncode == 0


def test_no_limit_is_raised_once_per_process():
    """Every kernel that asks for more than the default goes through SharedLimit."""
    for name in sorted(os.listdir(CSRC)):
        text = open(os.path.join(CSRC, name)).read()
        if name != "ddflb_smem.h":
            assert "cudaFuncSetAttribute(" not in text, name
