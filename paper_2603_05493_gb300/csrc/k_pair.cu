// k_pair.cu -- the single-robot pair kernel: one warp per configuration,
// persistent grid; the per-configuration work is pair_one_culled (default)
// or the full map-reduce pair_one (pair_body.cuh).
#include "pair_body.cuh"

#include <algorithm>

namespace wbe {

template <bool FULL, bool BITS, bool CULL>
__device__ __forceinline__ void pair_warps(const DevRobot& r, const PairSchedule32& ps,
                                           const FwdArgs& A) {
  extern __shared__ __align__(128) float smem[];
  const PairPlan pl(r.n, r.Sg, r.P, BITS, !CULL);
  float4* radw = reinterpret_cast<float4*>(smem);
  for (int i = threadIdx.x; i < r.Sg; i += blockDim.x) radw[i] = __ldg(r.grp_rad + i);
  __syncthreads();
  const int lane = threadIdx.x & 31;
  const int warp = threadIdx.x >> 5;
  const int wpb = blockDim.x >> 5;
  float* ws = smem + a32(4 * r.Sg) + warp * pl.total;
  for (int64_t b = (int64_t)blockIdx.x * wpb + warp; b < A.B; b += (int64_t)gridDim.x * wpb)
    if (CULL)
      pair_one_culled<FULL, BITS>(r, ps, A, b, ws, radw, lane);
    else
      pair_one<FULL, BITS>(r, ps, A, b, ws, radw, lane);
}

// The culled map-reduce is capped at 72 registers: 7 blocks of 4 warps then
// fit an SM's registers, and its shared memory holds 7 (the humanoid's culled
// pair stage: 0.162 ms at 79 registers and 6 blocks, 0.155 ms at 72 and 7,
// without spills).  The full map-reduce keeps its own allocation (it would
// spill at 72).
template <bool FULL, bool BITS>
__global__ void __maxnreg__(72) pair_kernel(DevRobot r, PairSchedule32 ps, FwdArgs A) {
  pair_warps<FULL, BITS, true>(r, ps, A);
}
template <bool FULL, bool BITS>
__global__ void __launch_bounds__(256, 3) pair_full_kernel(DevRobot r, PairSchedule32 ps,
                                                          FwdArgs A) {
  pair_warps<FULL, BITS, false>(r, ps, A);
}

// Small robots (at most kThreadMaxS spheres and kThreadMaxP pairs, e.g. a
// 7-DoF arm: 28 spheres, 240 pairs): one thread per configuration.  A warp per
// configuration leaves most lanes idle on so few blocks, and its per-
// configuration staging and reductions cost more than the pairs.  Each thread
// places its configuration's spheres from its link poses into its column of
// shared memory ([3][S][threads]: a warp reads 32 consecutive words) and
// evaluates every masked pair exactly, in index order (the column stride is
// threads + 1, so that the warp's transposed output copy, which reads one
// configuration's centres across the lanes, hits distinct banks):
//   d = sqrt(|c_i - c_j|^2) - (r_i + r_j), kept when strictly smaller,
// the same arithmetic as the warp kernel's exact path and the same tie rule
// (smallest pair index), so the results are the same bits.  The sphere and
// pair tables are staged once per block.
constexpr int kThreadMaxS = 32, kThreadMaxP = 1024, kThreadBlock = 128;
bool pair_thread_ok(const DevRobot& r) { return r.S <= kThreadMaxS && r.P <= kThreadMaxP; }
static size_t pair_thread_smem(const DevRobot& r) {
  return 16 * (size_t)r.S + 16 * (size_t)r.P + 4 * (size_t)r.S +
         sizeof(float) * 3 * (size_t)r.S * (kThreadBlock + 1);
}

template <bool BITS>
__global__ void __launch_bounds__(kThreadBlock) pair_thread_kernel(DevRobot r, FwdArgs A) {
  extern __shared__ __align__(16) float sm[];
  const int S = r.S, P = r.P, n = r.n, t = threadIdx.x;
  const int T = blockDim.x + 1;  // column stride of the centres
  float4* sp = reinterpret_cast<float4*>(sm);  // [S] centre in the link frame, radius
  // [P] pairs, row-major sorted: the two spheres' column offsets (s T) and
  // their radius sum r_i + r_j
  int4* pr = reinterpret_cast<int4*>(sp + S);
  int* sl = reinterpret_cast<int*>(pr + P);    // [S] link of each sphere
  float* cs = reinterpret_cast<float*>(sl + S);  // [3][S][T] this block's sphere centres
  for (int i = t; i < S; i += blockDim.x) {
    sp[i] = __ldg(r.sph + i);
    sl[i] = __ldg(r.sph_link + i);
  }
  for (int i = t; i < P; i += blockDim.x) {
    const int2 ij = __ldg(r.pairs + i);
    const float rr = __ldg(r.sph + ij.x).w + __ldg(r.sph + ij.y).w;
    pr[i] = make_int4(ij.x * T, ij.y * T, __float_as_int(rr), 0);
  }
  __syncthreads();
  const int64_t b = (int64_t)blockIdx.x * blockDim.x + t;
  const int lane = t & 31;
  const int64_t b0 = b - lane;  // the warp's first configuration
  const int nw = A.B - b0 < 32 ? (int)(A.B - b0) : 32;  // configurations of this warp
  if (b0 >= A.B) return;
  float* cx = cs + t;
  float* cy = cs + (size_t)S * T + t;
  float* cz = cs + 2 * (size_t)S * T + t;
  const float4* poses = reinterpret_cast<const float4*>(A.pose + b * (int64_t)n * 12);
  int cur = -1;
  float Pw[12];
  for (int s = 0; s < S && lane < nw; ++s) {
    const int l = sl[s];
    if (l != cur) {  // the spheres of a link are consecutive in most robots
      const float4 x0 = __ldg(poses + 3 * l), x1 = __ldg(poses + 3 * l + 1),
                   x2 = __ldg(poses + 3 * l + 2);
      Pw[0] = x0.x; Pw[1] = x0.y; Pw[2] = x0.z; Pw[3] = x0.w;
      Pw[4] = x1.x; Pw[5] = x1.y; Pw[6] = x1.z; Pw[7] = x1.w;
      Pw[8] = x2.x; Pw[9] = x2.y; Pw[10] = x2.z; Pw[11] = x2.w;
      cur = l;
    }
    const float4 q = sp[s];
    const float cl[3] = {q.x, q.y, q.z};
    float c[3];
    rot(Pw, cl, c);
    c[0] += Pw[9];
    c[1] += Pw[10];
    c[2] += Pw[11];
    cx[(size_t)s * T] = c[0];
    cy[(size_t)s * T] = c[1];
    cz[(size_t)s * T] = c[2];
  }
  __syncwarp();
  if (A.sph) {  // the warp's configurations are one contiguous [nw][S][3] region
    const float* cw = cs + (t - lane);  // column of the warp's first configuration
    float* o = A.sph + b0 * S * 3;
    for (int c = 0; c < nw; ++c)
      for (int e = lane; e < 3 * S; e += 32) {
        const int sph = e / 3, k = e - 3 * sph;
        o[(size_t)c * 3 * S + e] = cw[((size_t)k * S + sph) * T + c];
      }
  }
  if (lane >= nw) return;
  if (!A.dmin && !BITS) return;
  float best = __int_as_float(0x7f800000);
  int bi = -1;
  uint32_t word = 0u;
  const int W = (P + 31) >> 5;
  for (int p = 0; p < P; ++p) {
    const int4 ij = pr[p];
    const float d = sqrtf(dist2(cx[ij.x], cy[ij.x], cz[ij.x], cx[ij.y], cy[ij.y], cz[ij.y])) -
                    __int_as_float(ij.z);
    if (d < best) {
      best = d;
      bi = p;
    }
    if (BITS) {
      word |= (d < 0.0f ? 1u : 0u) << (p & 31);
      if ((p & 31) == 31 || p == P - 1) {
        A.bits[b * (int64_t)W + (p >> 5)] = word;
        word = 0u;
      }
    }
  }
  if (A.dmin) {
    A.dmin[b] = best;
    A.worst[b] = bi;
    if (A.wdiff) {
      float dd[3] = {0.0f, 0.0f, 0.0f};
      if (bi >= 0) {
        const int4 ij = pr[bi];
        dd[0] = cx[ij.x] - cx[ij.y];
        dd[1] = cy[ij.x] - cy[ij.y];
        dd[2] = cz[ij.x] - cz[ij.y];
      }
      A.wdiff[3 * b] = dd[0];
      A.wdiff[3 * b + 1] = dd[1];
      A.wdiff[3 * b + 2] = dd[2];
    }
  }
}

// The same small robots when every group of 4 spheres lies on one link
// (sph_vec4) and no pair bits are wanted: 8 lanes a configuration, 4
// configurations a warp.  Lane g places group g from its link's pose (48
// contiguous bytes a lane, the configuration's row contiguous over the 8),
// keeps the group's constants in registers and writes its centres as float4
// rows; then the lanes share the 4x4 blocks, 16 distances for six 16-byte
// shared loads where the thread-per-configuration loop takes six 4-byte loads
// and a table entry a pair.  The distances use the approximate square root:
// each lane keeps the least, its pair and the second least, the 8 lanes meet
// in shuffles, and the winner's distance is computed exactly.  When the second
// least is within the approximation's margin of the least (or anything is not
// a number), the configuration's pairs are evaluated exactly in index order,
// so the result is the exact path's, bit for bit, ties included.  Bound by
// issue (16 instructions a pair).  7-DoF arm: 0.064 -> 0.039 ms at 131072
// configurations, 0.023 -> 0.004 ms at 3300, 0.026 -> 0.004 ms at 64, where one
// thread's 240 serial pairs were the time.
constexpr int kSmallWarps = 8;
constexpr int kSmallGroups = kThreadMaxS / 4;
static bool pair_small_ok(const DevRobot& r, const FwdArgs& a) {
  return pair_thread_ok(r) && r.sph_vec4 && !a.bits;
}
static size_t pair_small_smem(const DevRobot& r) {
  return sizeof(float4) * kSmallGroups + sizeof(uint2) * (size_t)((r.nblk + 1) & ~1) +
         sizeof(float4) * kSmallWarps * 4 * 3 * kSmallGroups;
}

template <bool FULL>
__global__ void __launch_bounds__(32 * kSmallWarps) pair_small_kernel(
    const __grid_constant__ DevRobot r, const __grid_constant__ PairSchedule32 ps,
    const __grid_constant__ FwdArgs A) {
  extern __shared__ __align__(16) float4 smf[];
  constexpr int NG = kSmallGroups;
  float4* rad = smf;                                    // [NG] radii of each group
  uint2* blk = reinterpret_cast<uint2*>(smf + NG);      // [nblk] groups i | j << 16, mask
  const int nblk = r.nblk, Sg = r.Sg, S = r.S, n = r.n;
  for (int i = threadIdx.x; i < Sg; i += blockDim.x) rad[i] = __ldg(r.grp_rad + i);
  for (int i = threadIdx.x; i < 32 * ps.rounds; i += blockDim.x) {
    const uint2 e = __ldg(ps.ent + i);  // byte offsets 16 gi | 16 gj << 16, mask << 16 | block
    if ((e.y >> 16) != 0u) blk[e.y & 0xFFFF] = make_uint2((e.x >> 4) & 0x0FFF0FFFu, e.y >> 16);
  }
  __syncthreads();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, c = lane >> 3, l = lane & 7;
  // this configuration's centres: [3][NG] float4
  float4* C = smf + NG + (nblk + 1) / 2 + (warp * 4 + c) * 3 * NG;
  const float* Cf = reinterpret_cast<const float*>(C);
  const float* radf = reinterpret_cast<const float*>(rad);
  const bool has = l < Sg;
  const int link = has ? __ldg(r.grp_link + l) : 0;
  float4 sp[4];
#pragma unroll
  for (int q = 0; q < 4; ++q) sp[q] = has ? __ldg(r.sph + 4 * l + q) : make_float4(0, 0, 0, 0);
  const float inf = __int_as_float(0x7f800000);
  const bool so4 = (reinterpret_cast<uintptr_t>(A.sph) & 15u) == 0;
  const int64_t step = (int64_t)gridDim.x * kSmallWarps * 4;
  for (int64_t b0 = ((int64_t)blockIdx.x * kSmallWarps + warp) * 4; b0 < A.B; b0 += step) {
    const bool act = b0 + c < A.B;
    const int64_t b = act ? b0 + c : A.B - 1;
    if (has) {
      const float4* P4 = reinterpret_cast<const float4*>(A.pose + (b * n + link) * 12);
      const float4 t0 = __ldg(P4), t1 = __ldg(P4 + 1), t2 = __ldg(P4 + 2);
      const float T[12] = {t0.x, t0.y, t0.z, t0.w, t1.x, t1.y, t1.z, t1.w, t2.x, t2.y, t2.z, t2.w};
      float o[12];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const float cl[3] = {sp[q].x, sp[q].y, sp[q].z};
        rot(T, cl, o + 3 * q);
#pragma unroll
        for (int i = 0; i < 3; ++i) o[3 * q + i] += T[9 + i];
      }
      C[l] = make_float4(o[0], o[3], o[6], o[9]);
      C[NG + l] = make_float4(o[1], o[4], o[7], o[10]);
      C[2 * NG + l] = make_float4(o[2], o[5], o[8], o[11]);
      if (A.sph && act) {
        float* so = A.sph + (b * S + 4 * l) * 3;
        if (so4) {
          float4* o4 = reinterpret_cast<float4*>(so);
          o4[0] = make_float4(o[0], o[1], o[2], o[3]);
          o4[1] = make_float4(o[4], o[5], o[6], o[7]);
          o4[2] = make_float4(o[8], o[9], o[10], o[11]);
        } else {
#pragma unroll
          for (int i = 0; i < 12; ++i) so[i] = o[i];
        }
      }
    }
    __syncwarp();
    if (A.dmin) {
      float m1 = inf, m2 = inf;  // least and second least approximate distance
      int at = 0;                // the least's slot in blk_pidx
      for (int k = l; k < nblk; k += 8) {
        const uint2 e = blk[k];
        const int gi = e.x & 0xFFFF, gj = e.x >> 16;
        const float4 xi = C[gi], yi = C[NG + gi], zi = C[2 * NG + gi], ri = rad[gi];
        const float4 xj = C[gj], yj = C[NG + gj], zj = C[2 * NG + gj], rj = rad[gj];
        const float ax[4] = {xi.x, xi.y, xi.z, xi.w}, ay[4] = {yi.x, yi.y, yi.z, yi.w},
                    az[4] = {zi.x, zi.y, zi.z, zi.w}, ar[4] = {ri.x, ri.y, ri.z, ri.w};
        const float bx[4] = {xj.x, xj.y, xj.z, xj.w}, by[4] = {yj.x, yj.y, yj.z, yj.w},
                    bz[4] = {zj.x, zj.y, zj.z, zj.w}, br[4] = {rj.x, rj.y, rj.z, rj.w};
#pragma unroll
        for (int t = 0; t < 16; ++t) {
          const int p = t >> 2, q = t & 3;
          float d = sqrt_approx(dist2(ax[p], ay[p], az[p], bx[q], by[q], bz[q])) - (ar[p] + br[q]);
          if (!FULL) d = (e.y >> t) & 1u ? d : inf;
          m2 = fminf(m2, fmaxf(m1, d));
          if (d < m1) {
            m1 = d;
            at = 16 * k + t;
          }
        }
      }
#pragma unroll
      for (int off = 4; off > 0; off >>= 1) {
        const float o1 = __shfl_xor_sync(0xffffffffu, m1, off);
        const float o2 = __shfl_xor_sync(0xffffffffu, m2, off);
        const int oa = __shfl_xor_sync(0xffffffffu, at, off);
        m2 = fminf(fmaxf(m1, o1), fminf(m2, o2));
        if (o1 < m1) {
          m1 = o1;
          at = oa;
        }
      }
      // exact distance of pair p, as the exact path of every pair kernel
      auto exact = [&](int2 ij) {
        return sqrtf(dist2(Cf[ij.x], Cf[4 * NG + ij.x], Cf[8 * NG + ij.x], Cf[ij.y],
                           Cf[4 * NG + ij.y], Cf[8 * NG + ij.y])) -
               (radf[ij.x] + radf[ij.y]);
      };
      // the approximation is within 3e-7 of the centre distance; the margin
      // covers it at both distances (a robot's reach, and poses far beyond it)
      bool close = !(m2 - m1 > fmaf(1e-6f, fabsf(m1), r.margin));
      float best = inf;
      int bi = -1;
      if (!close) {
        bi = __ldg(r.blk_pidx + at);
        best = exact(__ldg(r.pairs + bi));
      }
      if (__any_sync(0xffffffffu, close)) {
        float e = inf;
        int ei = INT_MAX;
        for (int p = l; p < r.P && close; p += 8) {
          const float d = exact(__ldg(r.pairs + p));
          if (d < e) {
            e = d;
            ei = p;
          }
        }
#pragma unroll
        for (int off = 4; off > 0; off >>= 1) {
          const float od = __shfl_xor_sync(0xffffffffu, e, off);
          const int oi = __shfl_xor_sync(0xffffffffu, ei, off);
          if (od < e || (od == e && oi < ei)) {
            e = od;
            ei = oi;
          }
        }
        if (close) {
          best = e;
          bi = ei == INT_MAX ? -1 : ei;
        }
      }
      if (l == 0 && act) {
        A.dmin[b] = best;
        A.worst[b] = bi;
        if (A.wdiff) pair_diff(r, A, b, bi, Cf, Cf + 4 * NG, Cf + 8 * NG);
      }
    }
    __syncwarp();  // the centres are the next configurations'
  }
}

// Whether the thread-per-configuration kernel is the faster one: estimates in us from
// both kernels at 9150 to 300000 configurations of 8 to 32 spheres and 1 to 336 pairs
// (within 20 %).  A warp of the eight-lane kernel takes 4 configurations, a fixed
// price and one more for every 8 blocks beyond the first 8; a thread of the other its
// spheres and pairs one after the other, for which its blocks, 128 configurations'
// centres each, have to be resident.  So the latter is the better one for a few pairs
// and a batch that fills the chip: two links, 16 pairs, 131072 configurations 11.9 us
// and 21.3; the arm with 16 pairs, 50000 12.3 and 16.9; with all 240 30.1 and 22.6.
static cudaError_t thread_better(const DevRobot& r, int64_t B, bool* out) {
  *out = false;
  if (B < 24576) return cudaSuccess;  // too few to fill the chip with threads
  const size_t smem = pair_thread_smem(r);
  int blocks = 0;
  cudaError_t e = allow_smem((const void*)pair_thread_kernel<false>, smem);
  if (e == cudaSuccess)
    e = max_blocks((const void*)pair_thread_kernel<false>, kThreadBlock, smem, &blocks);
  if (e != cudaSuccess || blocks < 1) return e;
  const float k = 1e-3f * (float)B, S = (float)r.S, P = (float)r.P;
  const int more = (r.nblk > 8 ? (r.nblk + 7) / 8 : 1) - 1;
  const float lanes = 4.5f + k * (0.125f + 0.0016f * S + 0.073f * (float)more);
  const int64_t wave = (int64_t)blocks * kThreadBlock * sm_count();
  const float waves = (float)((B + wave - 1) / wave);
  const float one = 5.0f + 0.11f * S + 0.075f * P;  // a wave's latency
  const float rate = 3.0f + k * (0.006f * S + 0.0012f * P);
  *out = std::max(waves * one, rate) * (0.85f + 0.15f * waves) < lanes;
  return cudaSuccess;
}

static cudaError_t launch_pair_small(const DevRobot& r, const PairSchedule32& ps, const FwdArgs& a,
                                     cudaStream_t s) {
  const size_t smem = pair_small_smem(r);
  auto kern = r.all_full ? pair_small_kernel<true> : pair_small_kernel<false>;
  // blocks of 32 configurations; past 16 a multiprocessor each block takes
  // several passes, evenly, so that its tables are staged once for them
  const int64_t need = (a.B + 4 * kSmallWarps - 1) / (4 * kSmallWarps);
  const int64_t most = 16 * (int64_t)sm_count(), passes = (need + most - 1) / most;
  kern<<<(unsigned)((need + passes - 1) / passes), 32 * kSmallWarps, smem, s>>>(r, ps, a);
  return cudaGetLastError();
}

static cudaError_t launch_pair_thread(const DevRobot& r, const FwdArgs& a, cudaStream_t s) {
  const size_t smem = pair_thread_smem(r);
  auto kern = a.bits ? pair_thread_kernel<true> : pair_thread_kernel<false>;
  cudaError_t e = allow_smem((const void*)kern, smem);
  if (e != cudaSuccess) return e;
  const int64_t grid = (a.B + kThreadBlock - 1) / kThreadBlock;
  kern<<<(unsigned)grid, kThreadBlock, smem, s>>>(r, a);
  return cudaGetLastError();
}

template <bool FULL, bool BITS, bool CULL>
static cudaError_t pair_launch_t(const DevRobot& r, const PairSchedule32& ps, const FwdArgs& a,
                                 int grid, int warps, size_t smem, cudaStream_t s, int* occ) {
  auto kern = CULL ? pair_kernel<FULL, BITS> : pair_full_kernel<FULL, BITS>;
  cudaError_t e = allow_smem((const void*)kern, smem);
  if (e != cudaSuccess) return e;
  if (occ) return max_blocks((const void*)kern, warps * 32, smem, occ);
  kern<<<grid, warps * 32, smem, s>>>(r, ps, a);
  return cudaGetLastError();
}

template <bool CULL>
static cudaError_t pair_dispatch_t(const DevRobot& r, const PairSchedule32& ps, const FwdArgs& a,
                                   int grid, int warps, cudaStream_t s, int* occ) {
  const bool bits = a.bits != nullptr;
  const size_t smem = pair_smem(r, warps, bits, !CULL);
  if (r.all_full) {
    return bits ? pair_launch_t<true, true, CULL>(r, ps, a, grid, warps, smem, s, occ)
                : pair_launch_t<true, false, CULL>(r, ps, a, grid, warps, smem, s, occ);
  }
  return bits ? pair_launch_t<false, true, CULL>(r, ps, a, grid, warps, smem, s, occ)
              : pair_launch_t<false, false, CULL>(r, ps, a, grid, warps, smem, s, occ);
}

static cudaError_t pair_dispatch(const DevRobot& r, const PairSchedule32& ps, const FwdArgs& a,
                                 int grid, int warps, cudaStream_t s, int* occ, bool cull) {
  return cull ? pair_dispatch_t<true>(r, ps, a, grid, warps, s, occ)
              : pair_dispatch_t<false>(r, ps, a, grid, warps, s, occ);
}

cudaError_t launch_pair(const DevRobot& r, const PairSchedule32& ps, const FwdArgs& a, int grid,
                        int warps, cudaStream_t s, bool cull) {
  if (cull && pair_small_ok(r, a)) {  // small robots
    bool thread = false;
    const cudaError_t e = thread_better(r, a.B, &thread);
    if (e != cudaSuccess) return e;
    return thread ? launch_pair_thread(r, a, s) : launch_pair_small(r, ps, a, s);
  }
  if (cull && pair_thread_ok(r)) return launch_pair_thread(r, a, s);
  return pair_dispatch(r, ps, a, grid, warps, s, nullptr, cull);
}

// what a launch may need at most (the full map-reduce's)
size_t pair_block_smem(const DevRobot& r, int warps, bool bits) {
  return pair_smem(r, warps, bits, true);
}

cudaError_t pair_max_blocks_per_sm(const DevRobot& r, int warps, bool bits, int* out) {
  FwdArgs a{};
  a.bits = bits ? reinterpret_cast<uint32_t*>(16) : nullptr;  // only selects the variant
  return pair_dispatch(r, PairSchedule32{}, a, 0, warps, nullptr, out, true);
}

}  // namespace wbe
