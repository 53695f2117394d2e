// k_kin.cu -- kinematic Jacobians of chosen links and the whole-body centre of
// mass with its Jacobian, from the world link poses the forward sweep wrote
// (the "second kernel" outputs of Sec. 6.1.1; the columns follow Alg. 2).
//
// One warp per configuration (persistent grid).  The warp stages the poses
// and, at every depth-first position, the link's mass moment m_k x_k =
// m_k p_k + R_k h_k (h_k = m_k c_k, payload point masses included in the
// compact inertia), kept as exclusive prefix sums over the depth-first order
// so that any subtree's moment is one difference.  A lane per joint j then walks the links the joint
// drives (connectedLinks of Alg. 2, several for a mimic joint):
//   Jacobian of target e: a driven link l contributes when it is an ancestor
//     of e or e itself -- an O(1) test on depth-first ranges (l's subtree is
//     the range [pos_l, end_l)) in place of Alg. 2's affects / linkChain
//     filters -- with m_l [w x (p_e - p_l); w] for a revolute joint
//     (w = R_l a_l) and m_l [R_l a_l; 0] for a prismatic one;
//   centre of mass: sum_k m_k x_k / M, and column j of its Jacobian
//     sum_l m_l (w x (S_l - M_l p_l)) / M (revolute) or M_l R_l a_l / M
//     (prismatic), with S_l and M_l the mass moment and mass of l's subtree:
//     the difference of the prefix sums at the ends of its contiguous
//     depth-first range.
// Rows of a link Jacobian: velocity of the world origin, then angular
// velocity, both in world coordinates.
#include "spatial.cuh"

namespace wbe {

// per warp: link poses, then the exclusive prefix sums of the mass moments
// over the depth-first order (n + 1 float4)
static __host__ __device__ int kin_words(int n) {
  return ((12 * n + 31) & ~31) + ((4 * (n + 1) + 31) & ~31);
}

__global__ void __launch_bounds__(256) kin_kernel(DevRobot r, const __grid_constant__ KinArgs A) {
  extern __shared__ __align__(16) float smem[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, wpb = blockDim.x >> 5;
  const int n = r.n, d = r.d;
  float* P = smem + (size_t)warp * kin_words(n);       // poses
  float4* mom = reinterpret_cast<float4*>(P + ((12 * n + 31) & ~31));  // by DFS position
  for (int64_t b = (int64_t)blockIdx.x * wpb + warp; b < A.B; b += (int64_t)gridDim.x * wpb) {
    const float4* src = reinterpret_cast<const float4*>(A.pose + b * (int64_t)n * 12);
    float4* dst = reinterpret_cast<float4*>(P);
    for (int i = lane; i < 3 * n; i += 32) dst[i] = __ldg(src + i);
    __syncwarp();
    const bool want_com = A.com || A.jac_com;
    float M = 0.0f;
    if (want_com) {
      // mass moments by DFS position and their exclusive prefix sums
      // mom[pos] = sum of the first pos moments (warp scans, 32 at a time):
      // a subtree is a DFS range [pos_l, end_l), so its moment is
      // mom[end_l] - mom[pos_l], and the whole body's is mom[n]
      float4 carry = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
      if (lane == 0) mom[0] = carry;
      for (int p0 = 0; p0 < n; p0 += 32) {
        const int pos = p0 + lane;
        float4 v = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        if (pos < n) {
          const int k = __ldg(r.dfs + pos).x;
          const float* I = r.inert + 10 * k;
          const float mk = __ldg(I), h[3] = {__ldg(I + 1), __ldg(I + 2), __ldg(I + 3)};
          const float* T = P + 12 * k;
          float Rh[3];
          rot(T, h, Rh);
          v = make_float4(fmaf(mk, T[9], Rh[0]), fmaf(mk, T[10], Rh[1]), fmaf(mk, T[11], Rh[2]),
                          mk);
        }
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {  // inclusive scan
          const float x = __shfl_up_sync(0xffffffffu, v.x, off);
          const float y = __shfl_up_sync(0xffffffffu, v.y, off);
          const float z = __shfl_up_sync(0xffffffffu, v.z, off);
          const float w = __shfl_up_sync(0xffffffffu, v.w, off);
          if (lane >= off) {
            v.x += x;
            v.y += y;
            v.z += z;
            v.w += w;
          }
        }
        if (pos < n)
          mom[pos + 1] = make_float4(carry.x + v.x, carry.y + v.y, carry.z + v.z, carry.w + v.w);
        carry.x += __shfl_sync(0xffffffffu, v.x, 31);
        carry.y += __shfl_sync(0xffffffffu, v.y, 31);
        carry.z += __shfl_sync(0xffffffffu, v.z, 31);
        carry.w += __shfl_sync(0xffffffffu, v.w, 31);
      }
      __syncwarp();
      const float4 tot = mom[n];
      M = tot.w;
      if (A.com && lane == 0) {
        const float iM = M > 0.0f ? 1.0f / M : 0.0f;
        A.com[3 * b] = tot.x * iM;
        A.com[3 * b + 1] = tot.y * iM;
        A.com[3 * b + 2] = tot.z * iM;
      }
    }
    for (int j = lane; j < d; j += 32) {
      const int l0 = __ldg(r.jl_start + j), l1 = __ldg(r.jl_start + j + 1);
      // centre-of-mass column
      if (A.jac_com) {
        float c[3] = {0.0f, 0.0f, 0.0f};
        for (int li = l0; li < l1; ++li) {
          const int l = __ldg(r.jl_links + li);
          const float* T = P + 12 * l;
          const float4 a4 = __ldg(reinterpret_cast<const float4*>(r.axis) + l);
          const float a[3] = {a4.x, a4.y, a4.z};
          float wv[3];
          rot(T, a, wv);  // R_l a_l
          const float mm = __ldg(reinterpret_cast<const float2*>(r.mimic) + l).x;
          const float4 hi = mom[__ldg(r.dfs_end + l)], lo = mom[__ldg(r.dfs_pos + l)];
          const float S[3] = {hi.x - lo.x, hi.y - lo.y, hi.z - lo.z};
          const float Ms = hi.w - lo.w;
          if (__ldg(r.jtype + l) == 1) {
            const float rel[3] = {fmaf(-Ms, T[9], S[0]), fmaf(-Ms, T[10], S[1]),
                                  fmaf(-Ms, T[11], S[2])};
            float cr[3];
            cross3(wv, rel, cr);
            for (int i = 0; i < 3; ++i) c[i] = fmaf(mm, cr[i], c[i]);
          } else if (__ldg(r.jtype + l) == 2) {
            for (int i = 0; i < 3; ++i) c[i] = fmaf(mm * Ms, wv[i], c[i]);
          }
        }
        const float iM = M > 0.0f ? 1.0f / M : 0.0f;
        for (int i = 0; i < 3; ++i) A.jac_com[(b * 3 + i) * d + j] = c[i] * iM;
      }
      // link Jacobians
      if (A.jac) {
        for (int t = 0; t < A.nt; ++t) {
          const int e = A.targets[t];
          const int pe = __ldg(r.dfs_pos + e);
          const float* Te = P + 12 * e;
          float col[6] = {0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f};
          for (int li = l0; li < l1; ++li) {
            const int l = __ldg(r.jl_links + li);
            if (pe < __ldg(r.dfs_pos + l) || pe >= __ldg(r.dfs_end + l)) continue;  // not on e's chain
            const float* T = P + 12 * l;
            const float4 a4 = __ldg(reinterpret_cast<const float4*>(r.axis) + l);
            const float a[3] = {a4.x, a4.y, a4.z};
            float wv[3];
            rot(T, a, wv);
            const float mm = __ldg(reinterpret_cast<const float2*>(r.mimic) + l).x;
            if (__ldg(r.jtype + l) == 1) {
              const float rel[3] = {Te[9] - T[9], Te[10] - T[10], Te[11] - T[11]};
              float cr[3];
              cross3(wv, rel, cr);
              for (int i = 0; i < 3; ++i) {
                col[i] = fmaf(mm, cr[i], col[i]);
                col[3 + i] = fmaf(mm, wv[i], col[3 + i]);
              }
            } else if (__ldg(r.jtype + l) == 2) {
              for (int i = 0; i < 3; ++i) col[i] = fmaf(mm, wv[i], col[i]);
            }
          }
          float* o = A.jac + ((b * A.nt + t) * 6) * (int64_t)d + j;
          for (int i = 0; i < 6; ++i) o[(int64_t)i * d] = col[i];
        }
      }
    }
    __syncwarp();  // shared arrays are reused by the next configuration
  }
}

// The same for robots whose joints drive one link each.  What a lane needs of
// its joints and links is the same for every configuration: it is staged once
// per block (each link's mass moment by DFS position; each joint's axis,
// multiplier, link, depth-first range, and a bit per target it moves), where the
// general kernel above walks the joint's link list and six index arrays in
// global memory for every configuration.  The next configuration's poses are
// copied into a second buffer while this one computes, and a link's pose is read
// as three 16-byte words (12-float rows hit four banks otherwise).  The same
// arithmetic in the same order: the same bits.  Bound by its output stores;
// humanoid, 4 targets, 20011 configurations: 0.037 -> 0.026 ms.
struct KinPlan {  // shared memory in 16-byte words
  int hm, ja, ji, jm, buf, per_warp;
  __host__ __device__ KinPlan(int n, int d) {
    hm = 0;                       // [n] h, m by DFS position
    ja = hm + n;                  // [d] axis, multiplier
    ji = ja + d;                  // [d] link | type << 8, first and last position; targets lo, hi
    jm = ji + d;                  // [n] link of each DFS position (ints)
    buf = jm + (n + 3) / 4;
    per_warp = 2 * 3 * n + n + 1;  // two pose buffers, the moments' prefix sums
  }
  __host__ __device__ size_t bytes(int warps) const {
    return sizeof(float4) * ((size_t)buf + (size_t)warps * per_warp);
  }
};

__device__ __forceinline__ void pose_of(const float4* P, int k, float* T) {
  const float4 x = P[3 * k], y = P[3 * k + 1], z = P[3 * k + 2];
  T[0] = x.x; T[1] = x.y; T[2] = x.z; T[3] = x.w;
  T[4] = y.x; T[5] = y.y; T[6] = y.z; T[7] = y.w;
  T[8] = z.x; T[9] = z.y; T[10] = z.z; T[11] = z.w;
}

__global__ void __launch_bounds__(256) kin_single_kernel(const __grid_constant__ DevRobot r,
                                                         const __grid_constant__ KinArgs A) {
  extern __shared__ __align__(16) float4 smk[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, wpb = blockDim.x >> 5;
  const int n = r.n, d = r.d, nt = A.jac ? A.nt : 0;
  const KinPlan pl(n, d);
  float4* hm = smk + pl.hm;
  float4* ja = smk + pl.ja;
  int4* ji = reinterpret_cast<int4*>(smk + pl.ji);
  int* kp = reinterpret_cast<int*>(smk + pl.jm);
  for (int i = threadIdx.x; i < n; i += blockDim.x) {
    const int k = __ldg(r.dfs + i).x;
    const float* I = r.inert + 10 * k;
    hm[i] = make_float4(__ldg(I + 1), __ldg(I + 2), __ldg(I + 3), __ldg(I));
    kp[i] = k;
  }
  for (int j = threadIdx.x; j < d; j += blockDim.x) {
    const int l = __ldg(r.jl_links + __ldg(r.jl_start + j));
    const float4 a4 = __ldg(reinterpret_cast<const float4*>(r.axis) + l);
    ja[j] = make_float4(a4.x, a4.y, a4.z, __ldg(reinterpret_cast<const float2*>(r.mimic) + l).x);
    const int lo = __ldg(r.dfs_pos + l), hi = __ldg(r.dfs_end + l);
    uint64_t moves = 0;  // bit t: l is target t's link or an ancestor of it
    for (int t = 0; t < nt; ++t) {
      const int pe = __ldg(r.dfs_pos + A.targets[t]);
      moves |= (uint64_t)(pe >= lo && pe < hi) << t;
    }
    ji[j] = make_int4(l | (int)__ldg(r.jtype + l) << 8, lo | hi << 16, (int)(uint32_t)moves,
                      (int)(uint32_t)(moves >> 32));
  }
  __syncthreads();
  float4* ws = smk + pl.buf + (size_t)warp * pl.per_warp;
  float4* mom = ws + 6 * n;  // exclusive prefix sums of the moments by DFS position
  const bool want_com = A.com || A.jac_com;
  const int64_t step = (int64_t)gridDim.x * wpb;
  auto fetch = [&](int64_t b, float4* dst) {
    if (b < A.B) {
      const float4* src = reinterpret_cast<const float4*>(A.pose + b * (int64_t)n * 12);
      for (int i = lane; i < 3 * n; i += 32) {
        const unsigned to = static_cast<unsigned>(__cvta_generic_to_shared(dst + i));
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(to), "l"(src + i) : "memory");
      }
    }
    asm volatile("cp.async.commit_group;");
  };
  int64_t b = (int64_t)blockIdx.x * wpb + warp;
  fetch(b, ws);
  for (int side = 0; b < A.B; b += step, side ^= 1) {
    const float4* P = ws + side * 3 * n;
    fetch(b + step, ws + (side ^ 1) * 3 * n);
    asm volatile("cp.async.wait_group 1;" ::: "memory");
    __syncwarp();
    float M = 0.0f;
    if (want_com) {
      float4 carry = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
      if (lane == 0) mom[0] = carry;
      for (int p0 = 0; p0 < n; p0 += 32) {
        const int pos = p0 + lane;
        float4 v = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        if (pos < n) {
          const float4 h4 = hm[pos];
          const float h[3] = {h4.x, h4.y, h4.z}, mk = h4.w;
          float T[12], Rh[3];
          pose_of(P, kp[pos], T);
          rot(T, h, Rh);
          v = make_float4(fmaf(mk, T[9], Rh[0]), fmaf(mk, T[10], Rh[1]), fmaf(mk, T[11], Rh[2]),
                          mk);
        }
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {  // inclusive scan
          const float x = __shfl_up_sync(0xffffffffu, v.x, off);
          const float y = __shfl_up_sync(0xffffffffu, v.y, off);
          const float z = __shfl_up_sync(0xffffffffu, v.z, off);
          const float w = __shfl_up_sync(0xffffffffu, v.w, off);
          if (lane >= off) {
            v.x += x;
            v.y += y;
            v.z += z;
            v.w += w;
          }
        }
        if (pos < n)
          mom[pos + 1] = make_float4(carry.x + v.x, carry.y + v.y, carry.z + v.z, carry.w + v.w);
        carry.x += __shfl_sync(0xffffffffu, v.x, 31);
        carry.y += __shfl_sync(0xffffffffu, v.y, 31);
        carry.z += __shfl_sync(0xffffffffu, v.z, 31);
        carry.w += __shfl_sync(0xffffffffu, v.w, 31);
      }
      __syncwarp();
      const float4 tot = mom[n];
      M = tot.w;
      if (A.com && lane == 0) {
        const float iM = M > 0.0f ? 1.0f / M : 0.0f;
        A.com[3 * b] = tot.x * iM;
        A.com[3 * b + 1] = tot.y * iM;
        A.com[3 * b + 2] = tot.z * iM;
      }
    }
    const float iM = M > 0.0f ? 1.0f / M : 0.0f;
    for (int j = lane; j < d; j += 32) {
      const int4 in = ji[j];
      const float4 a4 = ja[j];
      const int jt = in.x >> 8;
      const float a[3] = {a4.x, a4.y, a4.z}, mm = a4.w;
      float T[12], wv[3];
      pose_of(P, in.x & 0xFF, T);
      rot(T, a, wv);  // R_l a_l
      if (A.jac_com) {  // centre-of-mass column
        float c[3] = {0.0f, 0.0f, 0.0f};
        const float4 hi = mom[in.y >> 16], lo = mom[in.y & 0xFFFF];
        const float S[3] = {hi.x - lo.x, hi.y - lo.y, hi.z - lo.z};
        const float Ms = hi.w - lo.w;
        if (jt == 1) {
          const float rel[3] = {fmaf(-Ms, T[9], S[0]), fmaf(-Ms, T[10], S[1]),
                                fmaf(-Ms, T[11], S[2])};
          float cr[3];
          cross3(wv, rel, cr);
#pragma unroll
          for (int i = 0; i < 3; ++i) c[i] = fmaf(mm, cr[i], c[i]);
        } else if (jt == 2) {
#pragma unroll
          for (int i = 0; i < 3; ++i) c[i] = fmaf(mm * Ms, wv[i], c[i]);
        }
        float* o = A.jac_com + b * 3 * (int64_t)d + j;
#pragma unroll
        for (int i = 0; i < 3; ++i) o[i * d] = c[i] * iM;
      }
      float* o = A.jac + b * nt * 6 * (int64_t)d + j;
      for (int t = 0; t < nt; ++t, o += 6 * d) {  // link Jacobians
        const float4 E = P[3 * A.targets[t] + 2];  // y, z of its rotation, its origin in y z w
        float col[6] = {0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f};
        if ((t < 32 ? (uint32_t)in.z >> t : (uint32_t)in.w >> (t - 32)) & 1u) {
          if (jt == 1) {
            const float rel[3] = {E.y - T[9], E.z - T[10], E.w - T[11]};
            float cr[3];
            cross3(wv, rel, cr);
#pragma unroll
            for (int i = 0; i < 3; ++i) {
              col[i] = fmaf(mm, cr[i], col[i]);
              col[3 + i] = fmaf(mm, wv[i], col[3 + i]);
            }
          } else if (jt == 2) {
#pragma unroll
            for (int i = 0; i < 3; ++i) col[i] = fmaf(mm, wv[i], col[i]);
          }
        }
#pragma unroll
        for (int i = 0; i < 6; ++i) o[i * d] = col[i];
      }
    }
    __syncwarp();  // shared arrays are reused by the next configuration
  }
  asm volatile("cp.async.wait_group 0;" ::: "memory");
}

// whether the single-link kernel takes it: one warp's workspace fits a block
static bool kin_single_ok(const DevRobot& r) {
  return !r.mimic_shared && KinPlan(r.n, r.d).bytes(1) <= 227 * 1024;
}
static int kin_single_warps(const DevRobot& r, int warps) {
  while (warps > 1 && KinPlan(r.n, r.d).bytes(warps) > 227 * 1024) --warps;
  return warps;
}

size_t kin_smem_per_warp(const DevRobot& r) { return sizeof(float) * kin_words(r.n); }

// Which kernel a call takes and how many of its blocks an SM holds.  A block of the
// general kernel has `warps` warps; the single-link one's at most as many.  The
// tables cost a block about half a microsecond, which one or two outputs (targets,
// the centre of mass) of robots with a joint a lane repay only when a warp takes
// more than one or two configurations: 23-DoF, one target, 3000 configurations 3.5
// us by the general kernel and 4.0 by the other, 32768 12.5 and 11.8; two targets
// 4.2 and 4.4, 17.2 and 14.4; four targets 5.4 and 5.1 (48-DoF, one target: 4.8 and
// 4.8, 25.4 and 24.4).  A lone target that few joints move is little work but for the
// tables, which a joint that does not move it needs all the same: the base of the
// 23-DoF tree, 32768 configurations 10.6 and 11.6.
cudaError_t kin_shape(const DevRobot& r, const KinArgs& a, int warps, int num_sms, int movers,
                      bool* single, int* bps) {
  const size_t smem = sizeof(float) * kin_words(r.n) * warps;
  cudaError_t e = allow_smem((const void*)kin_kernel, smem);
  if (e == cudaSuccess) e = max_blocks((const void*)kin_kernel, warps * 32, smem, bps);
  if (e != cudaSuccess) return e;
  const int outputs = (a.jac ? a.nt : 0) + (a.com || a.jac_com ? 1 : 0);
  const int64_t resident = (int64_t)*bps * warps * num_sms;
  const int64_t few = r.d > 32 || outputs > 2 ? 0 : outputs == 2 ? resident : 2 * resident;
  const bool still = outputs == 1 && a.jac && 8 * movers <= r.d;
  *single = kin_single_ok(r) && !still && a.B > few;
  if (!*single) return cudaSuccess;
  const int w = kin_single_warps(r, warps);
  const size_t smem1 = KinPlan(r.n, r.d).bytes(w);
  e = allow_smem((const void*)kin_single_kernel, smem1);
  if (e != cudaSuccess) return e;
  return max_blocks((const void*)kin_single_kernel, w * 32, smem1, bps);
}

cudaError_t launch_kin(const DevRobot& r, const KinArgs& a, bool single, int grid, int warps,
                       cudaStream_t s) {
  if (single) {
    const int w = kin_single_warps(r, warps);
    kin_single_kernel<<<grid, w * 32, KinPlan(r.n, r.d).bytes(w), s>>>(r, a);
  } else {
    kin_kernel<<<grid, warps * 32, sizeof(float) * kin_words(r.n) * warps, s>>>(r, a);
  }
  return cudaGetLastError();
}

}  // namespace wbe
