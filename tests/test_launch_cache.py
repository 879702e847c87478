"""The launch facts that are kept per kernel and device, against a CUDA runtime that the test supplies: out of memory on
the host no C++ exception leaves them (they are looked up inside C entry points), the opt-in to shared memory only rises,
and a size that was dropped from the kept ones is looked up again."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include <cstdio>
#include <cstdlib>
#include <new>
#include "paper_1610_02132_b200/csrc/qsgd_common.cuh"

static bool no_memory = false;
static int opted = 0, lookups = 0, lowered = 0;
void* operator new(std::size_t n) {
  if (no_memory) throw std::bad_alloc();
  return std::malloc(n);
}
void operator delete(void* p) noexcept { std::free(p); }
void operator delete(void* p, std::size_t) noexcept { std::free(p); }

extern "C" {
cudaError_t cudaGetDevice(int* d) { *d = 0; return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr, int) { *v = 148; return cudaSuccess; }
cudaError_t cudaFuncSetAttribute(const void*, cudaFuncAttribute, int v) {
  if (v < opted) ++lowered;
  opted = v;
  return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessor(int* n, const void*, int, size_t smem) {
  ++lookups;
  *n = (int)(232448 / (smem + 1024));
  return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* n, const void* f, int t, size_t smem, unsigned) {
  return cudaOccupancyMaxActiveBlocksPerMultiprocessor(n, f, t, smem);
}
}

int main() {
  static qsgd::KernelSite site;
  const void* kernel = &site;
  no_memory = true;
  for (int pass = 0; pass < 2; ++pass)
    for (size_t smem = 1024; smem <= 64 * 1024; smem += 1024)
      for (int again = 0; again < 2; ++again) {
        int sms = 0, occ = 0;
        if (site.lookup_dynamic(kernel, 256, smem, &sms, &occ) != 0 || sms != 148 || occ != (int)(232448 / (smem + 1024))) return 1;
      }
  std::printf("%d %d %d\n", opted, lowered, lookups);
  return 0;
}
"""


def test_launch_facts_without_host_memory(tmp_path):
    src, exe = tmp_path / "launch_cache.cpp", tmp_path / "launch_cache"
    src.write_text(PROGRAM)
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    subprocess.check_call([os.environ.get("CXX", "g++"), "-std=c++17", "-O1", "-w", "-I", ROOT, "-I", os.path.join(cuda, "include"), str(src),
                           "-o", str(exe), "-lpthread"])
    run = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert run.returncode == 0, run.stderr
    opted, lowered, lookups = map(int, run.stdout.split())
    assert opted == 64 * 1024 and lowered == 0 and lookups == 2 * 64      # 64 sizes, more than are kept, each asked for twice
