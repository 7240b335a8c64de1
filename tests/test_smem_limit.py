"""The opt-in to more than 48 KB of dynamic shared memory is one kernel's on one device: the helper
of csrc/smem_limit.h against a fake CUDA runtime with several devices (host only), and no other
source file sets the attribute."""
import glob
import os
import subprocess

from paper_2409_18122_gb300 import build as B

PROGRAM = r"""
#include <stdio.h>
#include <string.h>
#include <thread>
#include <vector>
#include "smem_limit.h"

static thread_local int device = 0;
static std::atomic<int> calls[2][70];
static bool fail = false;
void a(int) {}
void b(int) {}   // the same signature as a
extern "C" cudaError_t cudaGetDevice(int* d) { *d = device; return cudaSuccess; }
extern "C" cudaError_t cudaFuncSetAttribute(const void* f, cudaFuncAttribute what, int v) {
  if (what != cudaFuncAttributeMaxDynamicSharedMemorySize || v != 60000) return cudaErrorInvalidValue;
  if (fail) return cudaErrorMemoryAllocation;
  ++calls[f == (const void*)b][device];
  return cudaSuccess;
}
int main() {
  fail = true;      // a failed call leaves nothing behind
  if (gs::allow_smem<a>(60000) != cudaErrorMemoryAllocation) return 1;
  fail = false;
  for (int round = 0; round < 3; ++round)
    for (device = 0; device < 70; ++device)
      if (gs::allow_smem<a>(60000) != cudaSuccess) return 2;
  std::vector<std::thread> ts;
  for (int t = 0; t < 8; ++t)
    ts.emplace_back([] { device = 3; for (int i = 0; i < 1000; ++i) gs::allow_smem<b>(60000); });
  for (auto& t : ts) t.join();
  for (int d = 0; d < 70; ++d) printf("%d ", (int)calls[0][d]);
  int other = 0;
  for (int d = 0; d < 70; ++d) other += d != 3 ? (int)calls[1][d] : 0;
  printf("| %d %d\n", (int)calls[1][3], other);
  return 0;
}
"""


def test_limit_is_kept_per_kernel_and_device(tmp_path):
    src, exe = tmp_path / "limit.cpp", tmp_path / "limit"
    src.write_text(PROGRAM)
    cuda = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(B.nvcc()))), "include")
    subprocess.check_call(["g++", "-std=c++17", "-pthread", "-I", B.CSRC, "-I", cuda, str(src), "-o", str(exe)])
    a, b = subprocess.check_output([str(exe)]).decode().split("|")
    assert [int(x) for x in a.split()] == [1] * 64 + [3] * 6     # once per device, always past the flags
    first, other = (int(x) for x in b.split())
    assert 1 <= first <= 8 and other == 0                        # threads that meet may each ask once


def test_the_attribute_is_set_in_one_place():
    users = [os.path.basename(f) for f in glob.glob(os.path.join(B.CSRC, "*")) if "cudaFuncSetAttribute(" in open(f).read()]
    assert users == ["smem_limit.h"]
