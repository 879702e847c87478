"""Kernels that put tables at places of their own in shared memory are only launched where their dynamic shared memory begins in
front of those: against a CUDA runtime that the test supplies."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include <cstdio>
#include <cstdlib>
#include "paper_1610_02132_b200/csrc/qsgd_common.cuh"

static int own = 0, lookups = 0;
extern "C" {
cudaError_t cudaGetDevice(int* d) { *d = 0; return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr which, int) {
  *v = which == cudaDevAttrReservedSharedMemoryPerBlock ? 1024 : 148;
  return cudaSuccess;
}
cudaError_t cudaFuncGetAttributes(cudaFuncAttributes* a, const void*) {
  ++lookups;
  *a = cudaFuncAttributes();
  a->sharedSizeBytes = (size_t)own;
  return cudaSuccess;
}
}

int main(int, char** argv) {
  static qsgd::KernelSite site;
  const void* kernel = &site;
  own = std::atoi(argv[1]);
  const int first = site.dynamic_begins_within(kernel, 2816), second = site.dynamic_begins_within(kernel, 2816);
  std::printf("%d %d %d\n", first, second, lookups);
  return 0;
}
"""


def test_dynamic_shared_memory_that_begins_too_late_is_refused(tmp_path):
    src, exe = tmp_path / "places.cpp", tmp_path / "places"
    src.write_text(PROGRAM)
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    subprocess.check_call([os.environ.get("CXX", "g++"), "-std=c++17", "-O1", "-w", "-I", ROOT, "-I", os.path.join(cuda, "include"), str(src),
                           "-o", str(exe), "-lpthread"])
    said = {own: subprocess.run([str(exe), str(own)], capture_output=True, text=True, timeout=60).stdout.split() for own in (0, 1792, 1793, 3000)}
    assert said[0] == said[1792] == ["0", "0", "1"]
    invalid = "9"                                          # cudaErrorInvalidConfiguration
    assert said[1793] == said[3000] == [invalid, invalid, "1"]
