// k_hinge.cu -- the all-pairs summed self-collision hinge with activation
// distance eta:
//   cost_b = w sum_p max(0, eta - d_p),  d_p = |c_i - c_j| - r_i - r_j
// over every masked pair, and its gradient on the sphere centres (a pair
// with d_p < eta adds -w u to dcost/dc_i and +w u to dcost/dc_j,
// u = (c_i - c_j) / |c_i - c_j|).  Feeding that gradient to the backward
// sweep as the sphere upstream gradient gives dcost/dq.
//
// One warp per configuration (a persistent grid beyond 4 passes).  The warp stages the
// configuration's link poses into shared memory, places its spheres (Sec.
// 6.1.1) as SoA rows and bounds every group of 4 with a sphere (C_g, R_g)
// (for a group on one link, the host-made sphere in its link frame moved
// with the link), as the pair stage does.  It then walks the pair stage's
// 4x4 block schedule: a block whose bound |C_i - C_j| - R_i - R_j (in halves,
// widened for their rounding) is at least eta holds no active pair.
// Each lane marks its surviving blocks of 32 rounds in a bit mask, the
// survivors are queued from a warp scan of the counts and worked 32 at a
// time, one block a lane, every masked pair exactly (sqrt distance).  A
// block's lane sums its pairs' cost and each of its 8 spheres' gradient in
// pair order; the row spheres' gradients, then (a second phase) the column
// spheres', go to a slot of shared memory and are added into the per-sphere
// gradient in a fixed order -- each group's slots by the lowest lane holding
// that group, in lane order -- and the lanes' costs meet in a fixed shuffle
// tree: no atomics, the same result on every run.
#include "spatial.cuh"

namespace wbe {

// per warp, 32-bit words: link poses while the spheres are placed, then the
// 32 block slots in the same region; the sphere SoA rows x, y, z, the group
// bounds (half_bound), the gradient SoA rows gx, gy, gz and the queue of
// surviving schedule entries
struct HingePlan {
  int xc, yc, zc, gb, gx, gy, gz, q, total;
  __host__ __device__ HingePlan(int n, int S) {
    const int s4 = (S + 3) & ~3, m = (s4 + 31) & ~31;
    const int p0 = (12 * n + 31) & ~31, ps = (32 * kSlotWords + 31) & ~31;
    const int p = p0 > ps ? p0 : ps;
    xc = p;
    yc = xc + m;
    zc = yc + m;
    gb = zc + m;
    q = gb + m;  // m >= 4 x groups; the queue behind the bounds, as the pair stage has it
    gx = q + 64;
    gy = gx + m;
    gz = gy + m;
    total = gz + m;
  }
  // a block's slot: the 12 gradient floats of its row spheres, then (a second
  // phase) of its column spheres (an odd stride: the lanes' writes hit
  // distinct banks)
  static constexpr int kSlotWords = 13;
};

size_t hinge_smem_per_warp(const DevRobot& r) {
  return sizeof(float) * HingePlan(r.n, r.S).total;
}
size_t hinge_smem_fixed(const DevRobot& r) { return sizeof(float) * ((4 * r.Sg + 31) & ~31); }
static size_t hinge_block_smem(const DevRobot& r, int warps) {
  return hinge_smem_fixed(r) + (size_t)warps * hinge_smem_per_warp(r);
}

__device__ __forceinline__ float4 ld4(const char* base, uint32_t off) {
  return *reinterpret_cast<const float4*>(base + off);
}
__device__ __forceinline__ float p4(const float4& v, int i) {
  return i == 0 ? v.x : (i == 1 ? v.y : (i == 2 ? v.z : v.w));
}

// 24 warps an SM (the slots share the pose region, so their workspaces fit):
// 80 registers a thread (against 16 warps at 122 registers: 0.337 -> 0.281 ms on
// the humanoid's 32768 configurations).
// FULL: every block holds all 16 pairs.
template <bool FULL>
__global__ void __launch_bounds__(128, 6) hinge_kernel(const __grid_constant__ DevRobot r,
                                                       const __grid_constant__ PairSchedule32 ps,
                                                       const __grid_constant__ HingeArgs A) {
  extern __shared__ __align__(16) float smem[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, wpb = blockDim.x >> 5;
  const int n = r.n, S = r.S, Sg = r.Sg;
  const HingePlan pl(n, S);
  float4* radw = reinterpret_cast<float4*>(smem);  // group radii, per block
  for (int i = threadIdx.x; i < Sg; i += blockDim.x) radw[i] = __ldg(r.grp_rad + i);
  __syncthreads();
  float* ws = smem + ((4 * Sg + 31) & ~31) + (size_t)warp * pl.total;
  float* P = ws;
  float *xc = ws + pl.xc, *yc = ws + pl.yc, *zc = ws + pl.zc;
  uint2* gb = reinterpret_cast<uint2*>(ws + pl.gb);
  float *gx = ws + pl.gx, *gy = ws + pl.gy, *gz = ws + pl.gz;
  float* slot = ws;  // over the poses, once the spheres are placed
  uint32_t* qu = reinterpret_cast<uint32_t*>(ws + pl.q);
  const char *cxc = reinterpret_cast<const char*>(xc), *cyc = reinterpret_cast<const char*>(yc),
             *czc = reinterpret_cast<const char*>(zc), *crad = reinterpret_cast<const char*>(radw),
             *cgb = reinterpret_cast<const char*>(gb);
  const float eta = A.eta, w = A.w;
  const int prs = ps.prs;
  constexpr int SW = HingePlan::kSlotWords;
  for (int64_t b = (int64_t)blockIdx.x * wpb + warp; b < A.B; b += (int64_t)gridDim.x * wpb) {
    {
      const float4* src = reinterpret_cast<const float4*>(A.pose + b * (int64_t)n * 12);
      float4* dst = reinterpret_cast<float4*>(P);
      for (int i = lane; i < 3 * n; i += 32) {  // asynchronous copies into shared memory
        const unsigned a = static_cast<unsigned>(__cvta_generic_to_shared(dst + i));
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(a), "l"(src + i) : "memory");
      }
      asm volatile("cp.async.commit_group;");
      asm volatile("cp.async.wait_group 0;" ::: "memory");
    }
    __syncwarp();
    // bounds relative to the first link, as in the pair stage
    const float ox = P[9], oy = P[10], oz = P[11];
    const float ow = fmaf(fabsf(ox) + fabsf(oy) + fabsf(oz), 1e-6f, 3e-6f);
    const float4 zero4 = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    if (lane == 0)  // the far sphere of the schedule's null blocks
      *reinterpret_cast<uint2*>(ws + pl.gb + far_words(Sg)) = far_bound();
    if (r.sph_vec4) {
      // every group of 4 on one link: a lane a group places its centres, its
      // bound and its gradient rows' zeros from one pose
      for (int g = lane; g < Sg; g += 32) {
        const float4* T4 = reinterpret_cast<const float4*>(P) + 3 * __ldg(r.grp_link + g);
        const float4 t0 = T4[0], t1 = T4[1], t2 = T4[2];
        const float T[12] = {t0.x, t0.y, t0.z, t0.w, t1.x, t1.y, t1.z, t1.w, t2.x, t2.y, t2.z, t2.w};
        const float4 lx = __ldg(r.sph_t + g), ly = __ldg(r.sph_t + Sg + g),
                     lz = __ldg(r.sph_t + 2 * Sg + g);
        const float px[4] = {lx.x, lx.y, lx.z, lx.w}, py[4] = {ly.x, ly.y, ly.z, ly.w},
                    pz[4] = {lz.x, lz.y, lz.z, lz.w};
        float cx[4], cy[4], cz[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const float cl[3] = {px[k], py[k], pz[k]};
          float c[3];
          rot(T, cl, c);
          cx[k] = c[0] + T[9];
          cy[k] = c[1] + T[10];
          cz[k] = c[2] + T[11];
        }
        reinterpret_cast<float4*>(xc)[g] = make_float4(cx[0], cx[1], cx[2], cx[3]);
        reinterpret_cast<float4*>(yc)[g] = make_float4(cy[0], cy[1], cy[2], cy[3]);
        reinterpret_cast<float4*>(zc)[g] = make_float4(cz[0], cz[1], cz[2], cz[3]);
        const float4 L = __ldg(r.grp_loc + g);
        const float cl[3] = {L.x, L.y, L.z};
        float c[3];
        rot(T, cl, c);
        const float scale = fabsf(T[9]) + fabsf(T[10]) + fabsf(T[11]) + fabsf(L.x) +
                            fabsf(L.y) + fabsf(L.z);
        gb[g] = half_bound(c[0] + T[9] - ox, c[1] + T[10] - oy, c[2] + T[11] - oz,
                           fmaf(scale, 1e-6f, fmaf(L.w, 1e-6f, L.w)) + ow);
        reinterpret_cast<float4*>(gx)[g] = zero4;
        reinterpret_cast<float4*>(gy)[g] = zero4;
        reinterpret_cast<float4*>(gz)[g] = zero4;
      }
    } else {
      for (int s = lane; s < 4 * Sg; s += 32) {
        float c[3] = {0.0f, 0.0f, 0.0f};  // padding: never in a masked pair
        if (s < S) {
          const float4 sp = __ldg(r.sph + s);
          const float* T = P + 12 * __ldg(r.sph_link + s);
          const float cl[3] = {sp.x, sp.y, sp.z};
          rot(T, cl, c);
          c[0] += T[9];
          c[1] += T[10];
          c[2] += T[11];
        }
        xc[s] = c[0];
        yc[s] = c[1];
        zc[s] = c[2];
      }
    }
    __syncwarp();
    for (int g = lane; g < Sg && !r.sph_vec4; g += 32) {  // the same for groups over several links
      const int gl = __ldg(r.grp_link + g);
      if (gl >= 0) {  // one link: its host-made bound, moved with the link
        const float4 L = __ldg(r.grp_loc + g);
        const float* T = P + 12 * gl;
        const float cl[3] = {L.x, L.y, L.z};
        float c[3];
        rot(T, cl, c);
        const float scale = fabsf(T[9]) + fabsf(T[10]) + fabsf(T[11]) + fabsf(L.x) +
                            fabsf(L.y) + fabsf(L.z);
        gb[g] = half_bound(c[0] + T[9] - ox, c[1] + T[10] - oy, c[2] + T[11] - oz,
                           fmaf(scale, 1e-6f, fmaf(L.w, 1e-6f, L.w)) + ow);
      } else {
        gb[g] = mixed_bound(reinterpret_cast<const float4*>(xc)[g], reinterpret_cast<const float4*>(yc)[g],
                            reinterpret_cast<const float4*>(zc)[g], radw[g], S - 4 * g, ox, oy, oz, ow);
      }
      reinterpret_cast<float4*>(gx)[g] = zero4;
      reinterpret_cast<float4*>(gy)[g] = zero4;
      reinterpret_cast<float4*>(gz)[g] = zero4;
    }
    __syncwarp();
    float cost = 0.0f;
    const uint2* off = ps.off + lane;
    uint2 en = __ldg(off);  // one step ahead (the table ends with a null row)
    for (int u0 = 0; u0 < prs; u0 += 16) {
      // blocks whose bound is under eta can hold an active pair; bit v: round
      // 2 (u0 + v), bit 16 + v: the one after
      uint32_t km = 0u;
      const int u1 = min(prs - u0, 16);
#pragma unroll 2
      for (int v = 0; v < u1; ++v) {
        const uint2 e = en;
        off += 32;
        en = __ldg(off);
        auto under = [&](uint32_t o) {  // also where the bound is no number
          return !(half_gap(*reinterpret_cast<const uint2*>(cgb + (o & 0xFFFF)),
                            *reinterpret_cast<const uint2*>(cgb + (o >> 16))) >= eta);
        };
        km |= (under(e.x) ? 1u << v : 0u) | (under(e.y) ? 0x10000u << v : 0u);
      }
      const int cnt = __popc(km);
      int sum = cnt;  // inclusive scan of the counts over the lanes
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int v = __shfl_up_sync(0xffffffffu, sum, o);
        if (lane >= o) sum += v;
      }
      const int tot = __shfl_sync(0xffffffffu, sum, 31);
      int pos = sum - cnt;
      for (int w0 = 0; w0 < tot; w0 += 32) {
        while (km && pos < w0 + 32) {
          qu[pos - w0] = (uint32_t)(32 * (__ffs(km) - 1) + lane);  // bit and lane
          km &= km - 1u;
          ++pos;
        }
        __syncwarp();
        const int count = min(32, tot - w0);
        // one block a lane: every masked pair exactly, in pair order.  A null entry
        // is here where its bound was under eta or no number: no block
        // (the entries' rounds are decoded here: the queue is filled by few lanes)
        const uint32_t c = qu[lane], bit = c >> 5;
        const uint32_t at = 2 * ((u0 + (bit & 15)) * 32 + (c & 31)) + (bit >> 4);
        const uint2 e = lane < count ? sched_at(ps, at) : make_uint2(0u, 0u);
        const bool block = (e.y >> 16) != 0u;
        uint32_t key = 0xFFFFFFFFu;  // no block
        float gr[12];  // the lane's block: its row spheres' gradients, then its columns'
        if (block) {
          const uint32_t ro = e.x & 0xFFFF, co = e.x >> 16, mask = e.y >> 16;
          key = e.x;
          const float4 XR = ld4(cxc, ro), YR = ld4(cyc, ro), ZR = ld4(czc, ro), RR = ld4(crad, ro);
          const float4 XC = ld4(cxc, co), YC = ld4(cyc, co), ZC = ld4(czc, co), RC = ld4(crad, co);
          float gc[12];
#pragma unroll
          for (int k = 0; k < 12; ++k) gr[k] = gc[k] = 0.0f;
#pragma unroll
          for (int t = 0; t < 16; ++t) {
            if (!FULL && !((mask >> t) & 1u)) continue;
            const int ia = t >> 2, jc = t & 3;
            const float dx = p4(XR, ia) - p4(XC, jc), dy = p4(YR, ia) - p4(YC, jc),
                        dz = p4(ZR, ia) - p4(ZC, jc);
            const float nrm = sqrtf(fmaf(dz, dz, fmaf(dy, dy, dx * dx)));
            const float d = nrm - (p4(RR, ia) + p4(RC, jc));
            if (d < eta) {
              cost = fmaf(w, eta - d, cost);
              if (nrm > 0.0f) {
                const float k = w / nrm;
                gr[3 * ia] = fmaf(-k, dx, gr[3 * ia]);
                gr[3 * ia + 1] = fmaf(-k, dy, gr[3 * ia + 1]);
                gr[3 * ia + 2] = fmaf(-k, dz, gr[3 * ia + 2]);
                gc[3 * jc] = fmaf(k, dx, gc[3 * jc]);
                gc[3 * jc + 1] = fmaf(k, dy, gc[3 * jc + 1]);
                gc[3 * jc + 2] = fmaf(k, dz, gc[3 * jc + 2]);
              }
            }
          }
          float* sl = slot + lane * SW;
#pragma unroll
          for (int k = 0; k < 12; ++k) sl[k] = gr[k];
#pragma unroll
          for (int k = 0; k < 12; ++k) gr[k] = gc[k];  // the column side, written next
        }
        // add the slots into the spheres' gradients: the row groups, then the
        // column groups, each group's slots by their lowest lane in lane order
        // (shared among the lanes that hold them, a component each, the sums were
        // slower: 0.091 -> 0.120 ms)
#pragma unroll
        for (int side = 0; side < 2; ++side) {
          if (side == 1 && block) {
            float* sl = slot + lane * SW;
#pragma unroll
            for (int k = 0; k < 12; ++k) sl[k] = gr[k];
          }
          __syncwarp();
          const uint32_t grp = side == 0 ? (key & 0xFFFFu) : (key >> 16);  // byte offset
          const uint32_t same = __match_any_sync(0xffffffffu, block ? grp : 0xFFFFFFFFu);
          if (block && (__ffs(same) - 1) == lane) {
            float4* X4 = reinterpret_cast<float4*>(reinterpret_cast<char*>(gx) + grp);
            float4* Y4 = reinterpret_cast<float4*>(reinterpret_cast<char*>(gy) + grp);
            float4* Z4 = reinterpret_cast<float4*>(reinterpret_cast<char*>(gz) + grp);
            float4 ax = *X4, ay = *Y4, az = *Z4;
            for (uint32_t m = same; m; m &= m - 1u) {
              const float* sl = slot + (__ffs(m) - 1) * SW;
              ax.x += sl[0]; ay.x += sl[1]; az.x += sl[2];
              ax.y += sl[3]; ay.y += sl[4]; az.y += sl[5];
              ax.z += sl[6]; ay.z += sl[7]; az.z += sl[8];
              ax.w += sl[9]; ay.w += sl[10]; az.w += sl[11];
            }
            *X4 = ax;
            *Y4 = ay;
            *Z4 = az;
          }
          __syncwarp();
        }
      }
    }
    if (A.g_sph) {  // [S][3] from the SoA gradient rows
      float* o = A.g_sph + b * (int64_t)S * 3;
      for (int e = lane; e < 3 * S; e += 32) {
        const int s = e / 3, k = e - 3 * s;
        o[e] = (k == 0 ? gx : k == 1 ? gy : gz)[s];
      }
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) cost += __shfl_xor_sync(0xffffffffu, cost, off);
    if (lane == 0 && A.cost) A.cost[b] = cost;
    __syncwarp();  // the shared arrays are reused by the next configuration
  }
}

static const void* hinge_of(const DevRobot& r) {
  return r.all_full ? (const void*)hinge_kernel<true> : (const void*)hinge_kernel<false>;
}

cudaError_t launch_hinge(const DevRobot& r, const PairSchedule32& ps, const HingeArgs& a, int grid,
                         int warps, cudaStream_t s) {
  const size_t smem = hinge_block_smem(r, warps);
  const cudaError_t e = allow_smem(hinge_of(r), smem);
  if (e != cudaSuccess) return e;
  if (r.all_full)
    hinge_kernel<true><<<grid, warps * 32, smem, s>>>(r, ps, a);
  else
    hinge_kernel<false><<<grid, warps * 32, smem, s>>>(r, ps, a);
  return cudaGetLastError();
}

cudaError_t hinge_max_blocks_per_sm(const DevRobot& r, int warps, int* out) {
  const size_t smem = hinge_block_smem(r, warps);
  const cudaError_t e = allow_smem(hinge_of(r), smem);
  if (e != cudaSuccess) return e;
  return max_blocks(hinge_of(r), warps * 32, smem, out);
}

}  // namespace wbe
