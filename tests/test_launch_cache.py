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


OCCUPANCY = r"""
#include "wbe_internal.h"
#include <cstdio>
static int g_pct = -1, g_asked = 0;
extern "C" {
cudaError_t cudaGetDevice(int* d) { *d = 0; return cudaSuccess; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr a, int) {
  *v = a == cudaDevAttrMaxRegistersPerMultiprocessor ? 65536
     : a == cudaDevAttrMaxThreadsPerMultiProcessor ? 2048
     : a == cudaDevAttrMaxBlocksPerMultiprocessor ? 32
     : a == cudaDevAttrReservedSharedMemoryPerBlock ? 1024 : 228 * 1024;
  return cudaSuccess;
}
cudaError_t cudaFuncGetAttributes(cudaFuncAttributes* f, const void*) {
  f->numRegs = 128;
  f->sharedSizeBytes = 0;
  return cudaSuccess;
}
cudaError_t cudaFuncSetAttribute(const void*, cudaFuncAttribute a, int v) {
  if (a == cudaFuncAttributePreferredSharedMemoryCarveout) g_pct = v;
  return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessor(int* n, const void*, int, size_t smem) {
  ++g_asked;
  *n = (int)((g_pct < 0 ? 100 : g_pct) * 228 * 1024 / 100 / (smem + 1024));
  return cudaSuccess;
}
}
int bad = 0;
#define EXPECT(x) if (!(x)) { std::printf("line %d: %s (carveout %d)\n", __LINE__, #x, g_pct); ++bad; }
int main() {
  const int k = 0, other = 0;
  using namespace wbe;
  int first = 0, n = 0;
  EXPECT(max_blocks(&other, 128, 18 * 1024, &first) == cudaSuccess && first == 12);
  EXPECT(g_pct == -1);  // a kernel without a preference keeps none
  fit_carveout(&k, 128, 3 * 1024);
  const int small = g_pct;
  EXPECT(small > 0 && small < 10);
  EXPECT(max_blocks(&k, 128, 18 * 1024, &n) == cudaSuccess && n == first);
  EXPECT(g_pct == small);
  fit_carveout(&k, 128, 18 * 1024);
  EXPECT(g_pct > small);
  launch_cache_clear(0);
  EXPECT(max_blocks(&k, 128, 18 * 1024, &n) == cudaSuccess && n == first);
  fit_carveout(&k, 128, 3 * 1024);
  EXPECT(g_pct == small);
  const int asked = g_asked;
  EXPECT(max_blocks(&k, 128, 18 * 1024, &n) == cudaSuccess && n == first && g_asked == asked);
  return bad;
}
"""


def test_occupancy_does_not_depend_on_earlier_launches(tmp_path):
    """The blocks an SM holds, asked after a launch of another shape has left its
    carveout: the same, and the carveout is put back."""
    run(tmp_path, OCCUPANCY)


def test_limit_is_only_raised(tmp_path):
    run(tmp_path, HARNESS)


def run(tmp_path, source):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    cuda = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc))), "include")
    if shutil.which("g++") is None or not os.path.exists(os.path.join(cuda, "cuda_runtime.h")):
        pytest.skip("needs g++ and the CUDA headers")
    main = tmp_path / "main.cpp"
    main.write_text(source)
    exe = str(tmp_path / "cache")
    subprocess.run(["g++", "-std=c++17", "-I" + CSRC, "-I" + cuda, str(main), "-x", "c++",
                    os.path.join(CSRC, "launch_cache.cu"), "-o", exe], check=True)
    r = subprocess.run([exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
