"""The kernels with more than 48 KB of dynamic shared memory are allowed it on
every device that launches them, and a refusal is reported: the helper of the
launchers against a runtime of two devices that remembers the limits."""
import os
import re
import shutil
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2609_09990_gb300", "csrc")

PROGRAM = r"""
#include "smem_limit.h"
static int device, limit[2] = {48 << 10, 48 << 10}, most = 227 << 10;
extern "C" cudaError_t cudaFuncSetAttribute(const void*, cudaFuncAttribute a, int v) {
  if (a != cudaFuncAttributeMaxDynamicSharedMemorySize || v > most) return cudaErrorInvalidValue;
  limit[device] = v;
  return cudaSuccess;
}
extern "C" cudaError_t cudaGetLastError() { return cudaSuccess; }
static void kernel(int) {}
static bool launch(int d, int bytes) { device = d; return gbd::allow_shared_memory(kernel, bytes) && bytes <= limit[d]; }
int main() {
  const int big = 170 << 10;
  return launch(0, big) && launch(1, big) && launch(0, big) && !launch(1, 300 << 10) && launch(1, big) ? 0 : 1;
}
"""


def test_every_device_is_allowed(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    inc = os.path.join(os.path.dirname(os.path.dirname(nvcc)), "include")
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-I" + inc, "-I" + CSRC, str(src), "-o", str(exe)], check=True)
    assert subprocess.run([str(exe)]).returncode == 0


def test_launchers_use_the_helper():
    for f in os.listdir(CSRC):
        text = open(os.path.join(CSRC, f)).read()
        launches = len(re.findall(r"cudaFuncSetAttribute\s*\(", text))
        assert launches == (1 if f == "smem_limit.h" else 0), f
