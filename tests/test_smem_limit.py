"""The dynamic shared memory a kernel is allowed, per device: the helper the
launchers use, against a stand-in for the two runtime calls that counts them
(compiled for the host; no GPU)."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SOURCE = r"""
#include "bm_smem.h"
#include <cstdio>
static int device = 0, calls[40];
extern "C" cudaError_t cudaGetDevice(int* d) { *d = device; return cudaSuccess; }
extern "C" cudaError_t cudaFuncSetAttribute(const void*, cudaFuncAttribute, int bytes) {
  if (bytes > 227 * 1024) return cudaErrorInvalidValue;
  ++calls[device];
  return cudaSuccess;
}
static void kernel() {}
int main() {
  std::atomic<unsigned> done{0};
  for (int r = 0; r < 3; ++r)
    for (device = 0; device < 40; ++device)
      if (bm::set_smem_once(kernel, 200 * 1024, done) != cudaSuccess) return 1;
  for (device = 0; device < 40; ++device) {
    if (calls[device] != (device < 32 ? 1 : 3)) return 2;
  }
  device = 1;  // a refused limit is not remembered as allowed
  std::atomic<unsigned> other{0};
  if (bm::set_smem_once(kernel, 228 * 1024, other) == cudaSuccess || other.load()) return 3;
  std::puts("ok");
}
"""


def test_limit_is_set_once_on_every_device(tmp_path):
    src, exe = tmp_path / "smem.cpp", tmp_path / "smem"
    src.write_text(SOURCE)
    csrc = os.path.join(ROOT, "paper_2609_00205_gb300", "csrc")
    subprocess.run(["g++", "-std=c++17", "-I", csrc, "-I", "/usr/local/cuda/include", str(src), "-o", str(exe)], check=True)
    assert subprocess.run([str(exe)], capture_output=True, text=True, check=True).stdout == "ok\n"


def test_line_kernels_set_the_limit_through_the_helper():
    """The line kernels' launchers keep no limit of their own per process."""
    with open(os.path.join(ROOT, "paper_2609_00205_gb300", "csrc", "bm_levels.cuh")) as f:
        text = f.read()
    assert text.count("set_smem_once(") == 2 and "cudaFuncSetAttribute" not in text
