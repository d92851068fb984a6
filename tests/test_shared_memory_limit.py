"""The shared-memory limit of a kernel is one value, whoever launches it.

The limit belongs to the function on its device.  Four threads that launch one
kernel with four sizes, each asking first (allow_smem of csrc/feti_smem.h),
run here against a runtime without a device: every launch must find a limit
that holds it.  No source sets the limit in another way.
"""
import os
import re
import subprocess

from fake_cuda import CSRC, cuda_include

PROGRAM = r"""
#include "feti_smem.h"
#include <atomic>
#include <thread>
#include <vector>

static std::atomic<int> limit{48 * 1024 - 1024};  // of the one kernel, with 1 KB of static arrays
static std::atomic<int> refused{0};
extern "C" {
cudaError_t cudaFuncGetAttributes(cudaFuncAttributes* a, const void*) {
  a->sharedSizeBytes = 1024;
  a->maxDynamicSharedSizeBytes = limit;
  return cudaSuccess;
}
cudaError_t cudaGetDevice(int* d) { *d = 0; return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr, int) { *v = 227 * 1024; return cudaSuccess; }
cudaError_t cudaFuncSetAttribute(const void*, cudaFuncAttribute, int v) {
  if (v + 1024 > 227 * 1024) return cudaErrorInvalidValue;
  limit = v;
  return cudaSuccess;
}
}
static void kernel() {}
int main() {
  std::vector<std::thread> t;
  for (int kb : {20, 50, 100, 226})
    t.emplace_back([kb] {
      for (int i = 0; i < 20000; ++i) {
        (void)feti::allow_smem(kernel, kb * 1024);
        std::this_thread::yield();
        if (kb * 1024 > limit) ++refused;
      }
    });
  for (auto& x : t) x.join();
  return refused ? 1 : 0;
}
"""


def test_concurrent_launches_of_different_sizes(tmp_path):
    src = tmp_path / "limit.cpp"
    src.write_text(PROGRAM)
    exe = str(tmp_path / "limit")
    subprocess.run(["g++", "-std=c++17", "-O1", str(src), "-o", exe, "-I", CSRC, "-I", cuda_include(),
                    "-I", "/usr/local/cuda/include", "-pthread"], check=True)
    assert subprocess.run([exe], timeout=120).returncode == 0


def test_only_one_place_sets_the_limit():
    users = [f for f in sorted(os.listdir(CSRC))
             if re.search(r"cudaFuncSetAttribute\s*\(", open(os.path.join(CSRC, f)).read())]
    assert users == ["feti_smem.h"]
