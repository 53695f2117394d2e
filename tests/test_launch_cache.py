"""The launchers' cache of runtime answers, against a fake runtime on the host: a
kernel's shared-memory limit is only ever raised, also by the calls after a robot
load has cleared the cache -- another thread may be about to launch with the
most -- and is raised again where a new context has lost it."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2603_05493_gb300", "csrc")

HARNESS = r"""
#include "wbe_internal.h"
#include <cstdio>
static int g_dev = 0, g_limit = 48 * 1024, g_sets = 0;
extern "C" {
cudaError_t cudaGetDevice(int* d) { *d = g_dev; return cudaSuccess; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr, int) { *v = 0; return cudaErrorUnknown; }
cudaError_t cudaFuncGetAttributes(cudaFuncAttributes*, const void*) { return cudaErrorUnknown; }
cudaError_t cudaFuncSetAttribute(const void*, cudaFuncAttribute a, int v) {
  if (a != cudaFuncAttributeMaxDynamicSharedMemorySize || v > 227 * 1024) return cudaErrorInvalidValue;
  g_limit = v;
  ++g_sets;
  return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessor(int* n, const void*, int, size_t smem) {
  *n = (int)smem <= g_limit ? 1 : 0;
  return cudaSuccess;
}
}
int bad = 0;
#define EXPECT(x) if (!(x)) { std::printf("line %d: %s (limit %d, sets %d)\n", __LINE__, #x, g_limit, g_sets); ++bad; }
int main() {
  const int k = 0;
  using namespace wbe;
  EXPECT(allow_smem(&k, 200 * 1024) == cudaSuccess && g_limit == 200 * 1024);
  EXPECT(allow_smem(&k, 60 * 1024) == cudaSuccess && g_limit == 200 * 1024 && g_sets == 1);
  launch_cache_clear(0);  // another thread loads a robot and makes a small call
  EXPECT(allow_smem(&k, 60 * 1024) == cudaSuccess);
  EXPECT(g_limit == 200 * 1024);  // the first thread's launch is still allowed
  int n = 0;
  EXPECT(max_blocks(&k, 128, 200 * 1024, &n) == cudaSuccess && n == 1);
  launch_cache_clear(0);
  g_limit = 48 * 1024;  // a new context
  EXPECT(allow_smem(&k, 100 * 1024) == cudaSuccess && g_limit >= 100 * 1024);
  EXPECT(allow_smem(&k, 210 * 1024) == cudaSuccess && g_limit == 210 * 1024);
  EXPECT(allow_smem(&k, 230 * 1024) != cudaSuccess && g_limit == 210 * 1024);
  EXPECT(allow_smem(&k, 210 * 1024) == cudaSuccess);
  return bad;
}
"""


def test_limit_is_only_raised(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    cuda = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc))), "include")
    if shutil.which("g++") is None or not os.path.exists(os.path.join(cuda, "cuda_runtime.h")):
        pytest.skip("needs g++ and the CUDA headers")
    main = tmp_path / "main.cpp"
    main.write_text(HARNESS)
    exe = str(tmp_path / "cache")
    subprocess.run(["g++", "-std=c++17", "-I" + CSRC, "-I" + cuda, str(main), "-x", "c++",
                    os.path.join(CSRC, "launch_cache.cu"), "-o", exe], check=True)
    r = subprocess.run([exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
