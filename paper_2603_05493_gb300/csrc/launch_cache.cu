// launch_cache.cu -- what the launchers ask of the CUDA runtime, kept per kernel
// and device: the shared-memory limit, the occupancy, the carveout.
#include "wbe_internal.h"

#include <algorithm>
#include <mutex>
#include <vector>

namespace wbe {

// The runtime's answers per kernel and device: four of these calls a launch
// (two attributes set, the kernel's attributes and the occupancy read) were a
// third of a small call's time in the library.
namespace {
struct KernelState {
  const void* kern;
  int dev;
  size_t smem = 0;        // dynamic shared memory it is allowed
  size_t most = 0;        // the most it ever was: no call may lower it
  int carveout = cudaSharedmemCarveoutDefault;  // the last preference set
  int regs = -1;          // registers a thread (-1: not read yet)
  size_t stat = 0;        // static shared memory
  struct Occ {
    int threads;
    size_t smem;
    int blocks;
  };
  std::vector<Occ> occ;   // at most kOcc shapes
};
constexpr size_t kOcc = 64;
std::mutex g_kern_mu;
std::vector<KernelState> g_kern;

KernelState& kernel_state(const void* kern, int dev) {  // g_kern_mu held
  for (KernelState& k : g_kern)
    if (k.kern == kern && k.dev == dev) return k;
  g_kern.push_back(KernelState{kern, dev});
  return g_kern.back();
}
}  // namespace

// A robot load asks everything again (the context may be a new one).  The limit is
// then set back to the most it was and not to what that call needs: another
// thread may stand between its allow_smem and its launch.
void launch_cache_clear(int device) {
  std::lock_guard<std::mutex> lock(g_kern_mu);
  for (KernelState& k : g_kern)
    if (k.dev == device) {
      const size_t most = k.most;
      k = KernelState{k.kern, k.dev};
      k.most = most;
    }
}

cudaError_t allow_smem(const void* kern, size_t smem) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  std::lock_guard<std::mutex> lock(g_kern_mu);
  KernelState& k = kernel_state(kern, dev);
  if (smem <= k.smem) return cudaSuccess;
  const size_t limit = std::max(smem, k.most);
  e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)limit);
  if (e == cudaSuccess) k.smem = k.most = limit;
  return e;
}

cudaError_t max_blocks(const void* kern, int threads, size_t smem, int* out) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  std::lock_guard<std::mutex> lock(g_kern_mu);
  KernelState& k = kernel_state(kern, dev);
  for (const KernelState::Occ& o : k.occ)
    if (o.threads == threads && o.smem == smem) {
      *out = o.blocks;
      return cudaSuccess;
    }
  // The answer counts a carveout that a launch of another shape has left (asked so,
  // the batch's forward of 48-DoF robots got a third of its blocks after one of
  // arms: 0.042 -> 0.062 ms): asked at the largest, which is what a launch that
  // needs it gets, and the preference put back.
  auto prefer = [&](int pct) {
    if (cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout, pct) !=
        cudaSuccess)
      cudaGetLastError();
  };
  prefer(cudaSharedmemCarveoutMaxShared);
  e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(out, kern, threads, smem);
  prefer(k.carveout);
  if (e != cudaSuccess) return e;
  if (k.occ.size() >= kOcc) k.occ.clear();
  k.occ.push_back({threads, smem, *out});
  return cudaSuccess;
}

// the SM limits fit_carveout needs, queried once per device (host threads may
// launch on several devices at once)
struct SmLimits {
  int smem_sm, regs_sm, threads_sm, blocks_sm, reserved, sms;
};
static bool sm_limits(int dev, SmLimits* out) {
  constexpr int kDevices = 64;
  static std::mutex mu;
  static SmLimits cache[kDevices];
  static bool have[kDevices] = {};
  auto query = [](int d, SmLimits* l) {
    return cudaDeviceGetAttribute(&l->regs_sm, cudaDevAttrMaxRegistersPerMultiprocessor, d) ==
               cudaSuccess &&
           cudaDeviceGetAttribute(&l->threads_sm, cudaDevAttrMaxThreadsPerMultiProcessor, d) ==
               cudaSuccess &&
           cudaDeviceGetAttribute(&l->blocks_sm, cudaDevAttrMaxBlocksPerMultiprocessor, d) ==
               cudaSuccess &&
           cudaDeviceGetAttribute(&l->sms, cudaDevAttrMultiProcessorCount, d) == cudaSuccess &&
           cudaDeviceGetAttribute(&l->reserved, cudaDevAttrReservedSharedMemoryPerBlock, d) ==
               cudaSuccess &&
           cudaDeviceGetAttribute(&l->smem_sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, d) ==
               cudaSuccess;
  };
  if (dev < 0 || dev >= kDevices) return query(dev, out);
  std::lock_guard<std::mutex> lock(mu);
  if (!have[dev]) {
    if (!query(dev, &cache[dev])) return false;
    have[dev] = true;
  }
  *out = cache[dev];
  return true;
}

int sm_count() {
  int dev = 0;
  SmLimits L;
  if (cudaGetDevice(&dev) == cudaSuccess && sm_limits(dev, &L) && L.sms > 0) return L.sms;
  cudaGetLastError();
  return 152;
}

// Shared memory and L1 are one array per SM.  Without a preference the
// driver gave the segmented sweeps, whose blocks hold 14-22 KB of partials, a
// 132 KB shared carveout (measured), and the L1 that caches their depth-first
// stacks shrank to match.  fit_carveout asks for the smallest carveout that
// still holds every block the registers, warps and block limit let one SM
// keep (a hint: the driver rounds it up to a carveout it supports).
void fit_carveout(const void* kern, int threads, size_t smem) {
  int dev = 0;
  SmLimits L;
  if (cudaGetDevice(&dev) != cudaSuccess || !sm_limits(dev, &L)) {
    cudaGetLastError();
    return;
  }
  std::lock_guard<std::mutex> lock(g_kern_mu);
  KernelState& k = kernel_state(kern, dev);
  if (k.regs < 0) {
    cudaFuncAttributes fa;
    if (cudaFuncGetAttributes(&fa, kern) != cudaSuccess) return;
    k.regs = fa.numRegs;
    k.stat = fa.sharedSizeBytes;
  }
  const int warps = (threads + 31) / 32;
  const int regs_warp = ((k.regs * 32 + 255) / 256) * 256;  // 256-register allocation unit
  int nb = std::min(L.threads_sm / (32 * warps), L.blocks_sm);
  if (regs_warp > 0) nb = std::min(nb, (L.regs_sm / regs_warp) / warps);
  const size_t per = smem + k.stat + (size_t)L.reserved;
  nb = std::min<int>(nb, (int)((size_t)L.smem_sm / per));
  const size_t need = (size_t)std::max(nb, 1) * per;
  const int pct = (int)std::min<size_t>(100, (need * 100 + L.smem_sm - 1) / L.smem_sm);
  if (pct == k.carveout) return;
  if (cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout, pct) ==
      cudaSuccess)
    k.carveout = pct;
  else
    cudaGetLastError();
}

}  // namespace wbe
