// tree_sweep.cuh -- one thread per configuration, one depth-first sweep over
// the kinematic tree (device functions shared by the single-robot and the
// batched kernels).
//
// The links are visited in depth-first pre-order (computed on the host).  A
// stack indexed by tree depth holds, for every ancestor of the current link,
// what its subtree still needs; when the sweep moves to a link of depth dep,
// every stack entry at depth >= dep belongs to a finished subtree and is
// closed ("post-order") before the new link is pushed.  All threads of a warp
// walk the same sequence, so control flow is uniform, joint-major I/O
// ([d][B]) is coalesced, and the stack (indexed by a warp-uniform depth)
// lives in coalesced, L1-cached local memory.  Every lane does useful work,
// which the level-synchronous schedule (a few links per level) cannot.
//
// Forward (Alg. 4): pre-order computes the local transform, the world pose
// (Sec. 6.1.1, written to link_pose), v_k, a_k and f_k = I a + v x* I v;
// post-order closes F_k = f_k + sum_children X_c^T F_c, emits
// tau_j += m_k S_k^T F_k and adds X_k^T F_k to the parent.
//
// Backward (the VJP of Alg. 4 and of FK; Alg. 5 and Alg. 1 give the
// structure): every pass of the adjoint fits the same sweep.  It is written in
// world axes about each link's own origin, with the Newton-Euler form of Alg. 4
// (angular velocity w, angular acceleration al, acceleration A of the origin;
// the origin's velocity cancels).  With the torque adjoints as joint rates,
// wb and ub are the links' angular and linear velocity of that virtual motion,
// and sum_j taubar_j tau_j = sum_k wb_k . n_k + ub_k . f_k.  s: the joint's
// world axis, r: the offset from the parent's origin.
//   pre-order:  W, w, al, A, wb, ub of the link from its parent's
//   post-order: the link's (n, f) and the gradients gw, gal, gA of wb . n +
//               ub . f (link_adjoint), its gradient wrench (Wn, Wf) of the
//               kinematic outputs, plus the children's sums; the joint's
//               gradients; the sums moved to the parent's origin:
//               qdd_bar = s . gal,  qd_bar = s . gw + (w x s) . gal
//               q_bar   = s . [Wn - w x gw - al x gal - A x gA - wb x n - ub x f]
//               gw_pa  += gw + qd s x gal + grad_w [gA . (w x (w x r))]
//               gal_pa += gal + r x gA,  gA_pa += gA
//               n_pa   += n + r x f,  f_pa += f,  Wn_pa += Wn + r x Wf
//               (revolute; the prismatic forms stand at the close)
// Derived from Alg. 4 by reverse-mode differentiation.  Against link axes with
// 6-vectors (24 floats of sums, a rotation of every vector at every link, up
// and down) the sums are 21 floats, a move between links is a few crosses, and
// nothing spills at the 128-register cap: humanoid48 backward 0.165 -> 0.138
// ms, with the cost and states from control points 0.131 -> 0.102 ms, the
// uneven batch's 0.234 -> 0.200 ms.  The sine and cosine are scaled to the
// unit circle (UNIT in local_xf_m): gradient error against 64 bits 3.5e-6 ->
// 1.0e-6 (humanoid, 32768 configurations), where without it the world
// rotations' drift from orthogonality gave 5.5e-6.  Storing the states of
// branching links and reloading them at their children's closes instead:
// 0.149 ms, 2.1e-6.  The forward keeps link axes: its torques feed the
// torque-limit hinges, and there the world form was no faster (0.079 and
// 0.077 ms).
//
// Segmented sweeps.  A tree with few links per level but many links in total
// leaves one thread per configuration with a long serial chain and, at a few
// tens of thousands of configurations, few warps per SM.  The DFS order can
// instead be cut into G contiguous segments, one warp per segment over the
// same 32 configurations.  The warp of segment g first replays the ancestors
// of its first link (pre-order data only; its own force,
// adjoint and wrench contributions are zero), then sweeps its links.  Every
// post-order quantity above is linear in the accumulated sums given the
// pre-order data, so the outputs of a link that several segments
// hold (an ancestor of a segment's first link) are the sums of the
// segments' partial outputs.  Those partials go to shared-memory slots and
// the kernel adds them in segment order (deterministic) after a barrier; all
// other outputs are written directly by the one segment that owns the link.
#pragma once

#include "spatial.cuh"
#include "spline_basis.cuh"

namespace wbe {

constexpr int TMAXD = 32;  // deepest tree the sweep kernels accept

// One segment of a segmented sweep (see above).  slot == nullptr: the whole
// DFS order, outputs written directly.
struct Seg {
  int p0, p1;          // DFS positions this segment owns
  int g, G;            // segment index, segments per configuration
  const int16_t* slot; // [n] shared output slot of a link or -1; nullptr = none
  float* part;         // partial outputs of this group: [nout][ns][G][32]
  int ns;              // shared slots
  int lane;
  // forward sweep with its force stack in shared memory: this thread's
  // entry 0, and the stride of the [depth][6][threads] layout (the block's
  // threads)
  float* fst = nullptr;
  int fstr = 0;
};

__device__ __forceinline__ Seg whole_sweep(const DevRobot& r) {
  return Seg{0, r.n, 0, 1, nullptr, nullptr, 0, 0};
}

// L2 prefetch hint for a global input of the next link, so that its DRAM
// latency overlaps the current link's arithmetic (measured on the 48-DoF
// humanoid: 11 % off the one-thread sweeps; an L1 hint gives the same).
// Only called on addresses inside the caller's buffers.
__device__ __forceinline__ void pf(const void* p) { asm volatile("prefetch.L2 [%0];" ::"l"(p)); }

// The joint states (q, qd, qdd of joint j) of the sweep's configuration b,
// from [d][B] arrays ...
struct ArrayStates {
  const float* q;
  const float* qd;
  const float* qdd;
  int64_t B, b;
  __device__ __forceinline__ float pos(int j) const { return __ldg(q + (int64_t)j * B + b); }
  __device__ __forceinline__ float vel(int j) const { return __ldg(qd + (int64_t)j * B + b); }
  __device__ __forceinline__ float acc(int j) const { return __ldg(qdd + (int64_t)j * B + b); }
  __device__ __forceinline__ void prefetch(int j, bool rates) const {
    pf(q + (int64_t)j * B + b);
    if (rates) {
      pf(qd + (int64_t)j * B + b);
      pf(qdd + (int64_t)j * B + b);
    }
  }
};

// ... or evaluated from uniform cubic B-spline control points (Sec. 4,
// Eq. bspline-cubic) where the sweep needs them: the configuration is sample
// s of trajectory tr, u points at that trajectory's first window knot of
// joint 0 (control points [d][K]) and bs at the sample's basis rows [3][4]
// (q, qd, qdd), computed once per configuration.  Same arithmetic as the
// B-spline forward kernel, so the states are the same bits.
struct SplineStates {
  const float* u;
  int K;
  const float* bs;
  __device__ __forceinline__ float row(int j, int r) const {
    const float* p = u + (int64_t)j * K;
    return bs_row(bs + 4 * r, __ldg(p), __ldg(p + 1), __ldg(p + 2), __ldg(p + 3));
  }
  __device__ __forceinline__ float pos(int j) const { return row(j, 0); }
  __device__ __forceinline__ float vel(int j) const { return row(j, 1); }
  __device__ __forceinline__ float acc(int j) const { return row(j, 2); }
  __device__ __forceinline__ void prefetch(int j, bool) const { pf(u + (int64_t)j * K); }
};

// where the partial output o of link k goes, or nullptr for a direct write
__device__ __forceinline__ float* seg_part(const Seg& sg, int k, int o) {
  if (!sg.slot) return nullptr;
  const int s = __ldg(sg.slot + k);
  if (s < 0) return nullptr;
  return sg.part + ((size_t)(o * sg.ns + s) * sg.G + sg.g) * 32 + sg.lane;
}

// c += a x b
__device__ __forceinline__ void cross3_acc(const float* a, const float* b, float* c) {
  c[0] = fmaf(a[1], b[2], fmaf(-a[2], b[1], c[0]));
  c[1] = fmaf(a[2], b[0], fmaf(-a[0], b[2], c[1]));
  c[2] = fmaf(a[0], b[1], fmaf(-a[1], b[0], c[2]));
}
// c -= a x b
__device__ __forceinline__ void cross3_sub(const float* a, const float* b, float* c) {
  c[0] = fmaf(-a[1], b[2], fmaf(a[2], b[1], c[0]));
  c[1] = fmaf(-a[2], b[0], fmaf(a[0], b[2], c[1]));
  c[2] = fmaf(-a[0], b[1], fmaf(a[1], b[0], c[2]));
}
// c += f a x (a x b) = f (a (a . b) - b (a . a)), f = 1 or -1
template <int SIGN>
__device__ __forceinline__ void centripetal_acc(const float* a, const float* b, float* c) {
  const float ab = SIGN * dot3(a, b), aa = SIGN * dot3(a, a);
#pragma unroll
  for (int i = 0; i < 3; ++i) c[i] = fmaf(-b[i], aa, fmaf(a[i], ab, c[i]));
}
// c += the gradient of g . (w x (w x b)) with respect to w: b (w . g) +
// g (w . b) - 2 w (b . g)
__device__ __forceinline__ void centripetal_grad(const float* w, const float* b, const float* g,
                                                 float* c) {
  const float wg = dot3(w, g), wb = dot3(w, b), bg = -2.0f * dot3(b, g);
#pragma unroll
  for (int i = 0; i < 3; ++i) c[i] = fmaf(w[i], bg, fmaf(g[i], wb, fmaf(b[i], wg, c[i])));
}

// Motion of a link from its parent's, all in world axes: angular velocity w,
// angular acceleration al and acceleration A of the link's origin, which sits
// r from the parent's; s: the joint's axis in the world, vq, aq its rate and
// acceleration (jt 1 revolute, 2 prismatic, 0 fixed).
__device__ __forceinline__ void joint_motion(int jt, const float* s, const float* r, float vq,
                                             float aq, const float* wp, const float* alp,
                                             const float* Ap, float* w, float* al, float* A) {
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    w[i] = wp[i];
    al[i] = alp[i];
    A[i] = Ap[i];
  }
  cross3_acc(alp, r, A);
  centripetal_acc<1>(wp, r, A);
  if (jt == 1) {
    const float sq[3] = {s[0] * vq, s[1] * vq, s[2] * vq};
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      w[i] += sq[i];
      al[i] = fmaf(s[i], aq, al[i]);
    }
    cross3_acc(wp, sq, al);
  } else if (jt == 2) {
    const float sq[3] = {2.0f * vq * s[0], 2.0f * vq * s[1], 2.0f * vq * s[2]};
#pragma unroll
    for (int i = 0; i < 3; ++i) A[i] = fmaf(s[i], aq, A[i]);
    cross3_acc(wp, sq, A);
  }
}

// y = Io x for the rotational part of the compact inertia
__device__ __forceinline__ void rot_inertia(const float* I, const float* x, float* y) {
  y[0] = fmaf(I[8], x[2], fmaf(I[7], x[1], I[4] * x[0]));
  y[1] = fmaf(I[9], x[2], fmaf(I[5], x[1], I[7] * x[0]));
  y[2] = fmaf(I[6], x[2], fmaf(I[9], x[1], I[8] * x[0]));
}

// world pose W = P o L (12 floats each); t: the offset of W's origin from P's
__device__ __forceinline__ void compose(const float* P, const float* L, float* W, float* t) {
  matmul3(P, L, W);
  rot(P, L + 9, t);
  W[9] = P[9] + t[0];
  W[10] = P[10] + t[1];
  W[11] = P[11] + t[2];
}

template <class St>
__device__ __forceinline__ void link_local_m(const DevRobot& r, int k, int meta, const St& st,
                                             float* L) {  // meta: lmeta[k]
  const int j = (meta & 0xFFFF) - 1;
  const float th = j >= 0 ? joint_var(r, k, st.pos(j)) : 0.0f;
  local_xf_m(r, k, th, (meta >> 16) & 0xFF, ((meta >> 24) & 1) != 0, L, L + 9);
}
template <class St>
__device__ __forceinline__ void link_local(const DevRobot& r, int k, const St& st, float* L) {
  const int j = __ldg(r.jidx + k);
  const float th = j >= 0 ? joint_var(r, k, st.pos(j)) : 0.0f;
  local_xf(r, k, th, L, L + 9);
}

// the dfs_kj word of link k, built from the per-link arrays (for the
// replayed ancestors of a segment, which are not at its DFS positions)
__device__ __forceinline__ int packed_link(const DevRobot& r, int k) {
  const int nch = min(__ldg(r.child_start + k + 1) - __ldg(r.child_start + k), 255);
  return (__ldg(r.lmeta + k) & 0xFFFF) | (nch << 16) | ((int)__ldg(r.jtype + k) << 24) |
         ((int)__ldg(r.rot_id + k) << 26);
}

// ---------------------------------------------------------------------------
// forward: FK + RNEA
// ---------------------------------------------------------------------------
// Per-depth stack entry.  The local transform is not kept: post-order
// recomputes it from q (cheaper than a round trip through local memory).
// W, v and a are read only by the push of a second or later child, so only
// links with two or more children store them; F (own force plus the
// children's) is stored when a child's push interrupts it.
struct FEnt {
  float W[12];  // world pose
  float v[6], a[6], F[6];
};

// FS: the accumulated forces F of the stack live in shared memory (sg.fst)
// instead of the thread's local stack
template <class St, bool FS = false>
__device__ __forceinline__ void tree_fwd_seg(const DevRobot& r, const FwdArgs& A, const St& st,
                                             int64_t b, const Seg& sg) {
  const int64_t B = A.B;
  const int n = r.n;
  const bool dyn = A.tau != nullptr;
  FEnt stk[TMAXD];
  if (dyn && r.mimic_shared)
    for (int j = 0; j < r.d; ++j) A.tau[(int64_t)j * B + b] = 0.0f;
  // Register copies that spare most stack loads: the pre-order data of the
  // last pushed entry (never changes while the entry is on the stack; a link
  // pushed right after its parent reads it from here), and the accumulated
  // force of the entry that the post-order closes next (an unwinding chain
  // passes it on in registers; it is stored when a push interrupts).
  float cW[12], cv[6], ca[6];
  int cdep = -1;
  float pF[6];
  int pdep = -1;
  int lastk = 0;  // last pushed link; the stack holds its ancestor chain
  int ck = 0;     // the link the next close takes

  auto close = [&](int e) {
    FEnt& E = stk[e];
    // the link at depth e: the last pushed one, then each closed link's
    // parent (one load off the critical path instead of two dependent ones
    // into the ancestor chains: humanoid48 forward 0.0934 -> 0.0892 ms; the
    // backward, at its register cap, spills more with it and is not faster)
    const int k = ck;
    ck = __ldg(r.parent + k);
    float F[6];
    if (pdep == e) {
#pragma unroll
      for (int i = 0; i < 6; ++i) F[i] = pF[i];
    } else {
#pragma unroll
      for (int i = 0; i < 6; ++i) F[i] = FS ? sg.fst[(6 * e + i) * sg.fstr] : E.F[i];
    }
    pdep = -1;
    const int meta = __ldg(r.lmeta + k);
    const int j = (meta & 0xFFFF) - 1;
    if (j >= 0) {
      const float4 a4 = ldp(reinterpret_cast<const float4*>(r.axis) + k);
      const float ax[3] = {a4.x, a4.y, a4.z};
      const float mm = ldp(reinterpret_cast<const float2*>(r.mimic) + k).x;
      const float t = mm * St_dot((meta >> 16) & 0xFF, ax, F);
      float* pt = seg_part(sg, k, 0);
      if (pt) {
        *pt = t;
      } else {
        float* dst = A.tau + (int64_t)j * B + b;
        *dst = r.mimic_shared ? *dst + t : t;
      }
    }
    if (e > 0) {
      float L[12], up[6];
      link_local_m(r, k, meta, st, L);
      xf_force_T(L, L + 9, F, up);
#pragma unroll
      for (int i = 0; i < 6; ++i)
        pF[i] = (FS ? sg.fst[(6 * (e - 1) + i) * sg.fstr] : stk[e - 1].F[i]) + up[i];
      pdep = e - 1;
    }
  };
  auto flush = [&]() {  // the pending force goes back to its stack entry
    if (pdep >= 0) {
#pragma unroll
      for (int i = 0; i < 6; ++i) {
        if (FS)
          sg.fst[(6 * pdep + i) * sg.fstr] = pF[i];
        else
          stk[pdep].F[i] = pF[i];
      }
      pdep = -1;
    }
  };

  // pre-order of link k at depth dep; own = false replays an ancestor of
  // the segment (pose, v, a only; no output, no force of its own); pre: the
  // joint states (pq, pqd, pqdd) were loaded ahead by the caller
  auto push = [&](int k, int dep, bool own, bool pre, float pq, float pqd, float pqdd, int ky) {
    const int jk = (ky & 0xFFFF) - 1, nch = (ky >> 16) & 0xFF, jtk = (ky >> 24) & 3;
    if (dyn) flush();  // the parent's force, when it is still pending
    FEnt& E = stk[dep];
    float L[12];
    {
      const float th = jk >= 0 ? joint_var(r, k, pre ? pq : st.pos(jk)) : 0.0f;
      local_xf_m(r, k, th, jtk, ((ky >> 26) & 1) != 0, L, L + 9);
    }
    float PW[12], vp[6], ap[6];
    if (dep > 0) {
      if (dep == cdep + 1) {
#pragma unroll
        for (int i = 0; i < 12; ++i) PW[i] = cW[i];
#pragma unroll
        for (int i = 0; i < 6; ++i) {
          vp[i] = cv[i];
          ap[i] = ca[i];
        }
      } else {
        const FEnt& P = stk[dep - 1];
#pragma unroll
        for (int i = 0; i < 12; ++i) PW[i] = P.W[i];
#pragma unroll
        for (int i = 0; i < 6; ++i) {
          vp[i] = P.v[i];
          ap[i] = P.a[i];
        }
      }
      float t[3];
      compose(PW, L, cW, t);
    } else {
#pragma unroll
      for (int i = 0; i < 12; ++i) cW[i] = L[i];
      vp[0] = vp[1] = vp[2] = vp[3] = vp[4] = vp[5] = 0.0f;
      ap[0] = ap[1] = ap[2] = 0.0f;
      ap[3] = r.abase[0];
      ap[4] = r.abase[1];
      ap[5] = r.abase[2];
    }
    cdep = dep;
    lastk = k;
    ck = k;
    if (nch > 1) {
#pragma unroll
      for (int i = 0; i < 12; ++i) E.W[i] = cW[i];
    }
    if (own && A.pose) {
      float4* dst = reinterpret_cast<float4*>(A.pose + (b * n + k) * 12);
      dst[0] = make_float4(cW[0], cW[1], cW[2], cW[3]);
      dst[1] = make_float4(cW[4], cW[5], cW[6], cW[7]);
      dst[2] = make_float4(cW[8], cW[9], cW[10], cW[11]);
    }
    if (dyn) {
      const int j = jk;
      const float4 a4 = ldp(reinterpret_cast<const float4*>(r.axis) + k);
      const float ax[3] = {a4.x, a4.y, a4.z};
      const float mm = ldp(reinterpret_cast<const float2*>(r.mimic) + k).x;
      const float vq = j >= 0 ? mm * (pre ? pqd : st.vel(j)) : 0.0f;
      const float aq = j >= 0 ? mm * (pre ? pqdd : st.acc(j)) : 0.0f;
      rnea_va(L, L + 9, vp, ap, jtk, ax, vq, aq, cv, ca);
      float F[6];
      if (own) {
        float I[10];
        load_inertia(r, k, I);
        rnea_force(I, cv, ca, F);
        if (A.fext) {  // f_k = I a + v x* I v - f_ext,k
          const float* fe = A.fext + (b * n + k) * 6;
#pragma unroll
          for (int i = 0; i < 6; ++i) F[i] -= __ldg(fe + i);
        }
      } else {
#pragma unroll
        for (int i = 0; i < 6; ++i) F[i] = 0.0f;
      }
      if (nch > 1) {
#pragma unroll
        for (int i = 0; i < 6; ++i) {
          E.v[i] = cv[i];
          E.a[i] = ca[i];
        }
      }
      // the force waits in the pending registers; a child's push stores it
#pragma unroll
      for (int i = 0; i < 6; ++i) pF[i] = F[i];
      pdep = dep;
    }
  };

  int sp = 0;
  if (sg.p0 > 0) {  // replay the proper ancestors of the first link
    const int k0 = __ldg(r.dfs + sg.p0).x;
    const int c0 = __ldg(r.chain_start + k0), c1 = __ldg(r.chain_start + k0 + 1);
    for (int c = c0; c < c1 - 1; ++c) {
      const int a = __ldg(r.chain + c);
      push(a, c - c0, false, false, 0.0f, 0.0f, 0.0f, packed_link(r, a));
    }
    sp = c1 - 1 - c0;
  }
  // The joint states of the link pushed next, loaded one link ahead into
  // registers, so that their latency overlaps the current link's closes and
  // push (measured on the 48-DoF humanoid at 2 segments x 448 threads:
  // 0.0985 -> 0.0970 ms against the L2 prefetch hint it replaces).
  float nq = 0.0f, nqd = 0.0f, nqdd = 0.0f;
  int2 nkd = sg.p0 < sg.p1 ? __ldg(r.dfs_kj + sg.p0) : make_int2(0, 0);
  {
    const int j0 = sg.p0 < sg.p1 ? (nkd.y & 0xFFFF) - 1 : -1;
    if (j0 >= 0) {
      nq = st.pos(j0);
      if (dyn) {
        nqd = st.vel(j0);
        nqdd = st.acc(j0);
      }
    }
  }
  for (int pos = sg.p0; pos < sg.p1; ++pos) {
    // link | depth << 8, (joint + 1) | children << 16 of this position: one
    // load for what the DFS order, the joint index and the child table gave
    // in four (humanoid48 forward 0.0898 -> 0.0885 ms), kept from the
    // previous step's look-ahead rather than loaded again (0.0844 -> 0.0835
    // ms; the backward, at its register cap, spills more with it: 0.1664 ->
    // 0.1684 ms)
    const int2 kd = nkd;
    const int k = kd.x & 0xFF, dep = (kd.x >> 8) & 0xFF;
    const float cq = nq, cqd = nqd, cqdd = nqdd;
    if (pos + 1 < sg.p1) {  // the next link's joint inputs
      nkd = __ldg(r.dfs_kj + pos + 1);
      const int jn = (nkd.y & 0xFFFF) - 1;
      if (jn >= 0) {
        nq = st.pos(jn);
        if (dyn) {
          nqd = st.vel(jn);
          nqdd = st.acc(jn);
        }
      }
    }
    if (dyn) {
      while (sp > dep) close(--sp);
      flush();
    }
    sp = dep + 1;
    push(k, dep, true, true, cq, cqd, cqdd, kd.y);
  }
  if (dyn) {
    while (sp > 0) close(--sp);
    flush();
  }
}

__device__ __forceinline__ void tree_fwd_one(const DevRobot& r, const FwdArgs& A, int64_t b) {
  tree_fwd_seg(r, A, ArrayStates{A.q, A.qd, A.qdd, A.B, b}, b, whole_sweep(r));
}

// ---------------------------------------------------------------------------
// backward: the whole adjoint in one sweep
// ---------------------------------------------------------------------------
// The close of a link needs the link's pre-order state (world pose W, w, al,
// A, wb, ub).  It does not come from a stack.  One state lives in registers:
// a push carries it down one link and a close carries it back up by undoing
// the same maps (w_pa = w - s qd, ...; W_pa = W L^-1), so a close reads no
// parent data at all, and the push of a later child finds its parent's state
// in the registers.  The rounding of the repeated maps and inverses drifts by
// a few float ulps per link visited.
// Per-depth stack entry, only what a later step reads:
//   tb  -- the link's torque adjoint m taubar, for a link with children (a
//          leaf's close follows its push and reads it from a register);
//   acc -- the children's sums of n, f, gw, gal, gA and the wrench, stored
//          only when the push of a sibling subtree interrupts them.
// The link's own terms are formed at its close from its state, and its
// gradient wrench of the kinematic outputs too (its world pose is in the
// registers there): nothing of the link's own travels through the stack.
constexpr int kSums = 21;   // n 3, f 3, gw 3, gal 3, gA 3, wrench 6
struct BEnt {
  float acc[kSums];
  float tb;
};

// world pose of link l by composing its ancestor chain (topology cache)
template <class St>
__device__ __forceinline__ void chain_pose(const DevRobot& r, int l, const St& st, float* P) {
  const int c0 = __ldg(r.chain_start + l), c1 = __ldg(r.chain_start + l + 1);
  for (int c = c0; c < c1; ++c) {
    float L[12];
    link_local(r, __ldg(r.chain + c), st, L);
    if (c == c0) {
#pragma unroll
      for (int i = 0; i < 12; ++i) P[i] = L[i];
    } else {
      float T[12], t[3];
      compose(P, L, T, t);
#pragma unroll
      for (int i = 0; i < 12; ++i) P[i] = T[i];
    }
  }
}

// parent pose from a link's world pose W and its local transform L: W L^-1;
// t: the offset of W's origin from the parent's
__device__ __forceinline__ void uncompose(const float* W, const float* L, float* P, float* t) {
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j)
      P[3 * i + j] =
          fmaf(W[3 * i + 2], L[3 * j + 2], fmaf(W[3 * i + 1], L[3 * j + 1], W[3 * i] * L[3 * j]));
  rot(P, L + 9, t);
  P[9] = W[9] - t[0];
  P[10] = W[10] - t[1];
  P[11] = W[11] - t[2];
}

// a point of a link (link coordinates sp) with gradient g adds the outer
// product g sp^T to the link's rotation gradient G (row-major) and g to that
// of its origin, f
__device__ __forceinline__ void point_grad(float4 sp, const float* g, float* G, float* f) {
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    G[3 * i] = fmaf(g[i], sp.x, G[3 * i]);
    G[3 * i + 1] = fmaf(g[i], sp.y, G[3 * i + 1]);
    G[3 * i + 2] = fmaf(g[i], sp.z, G[3 * i + 2]);
    f[i] += g[i];
  }
}

// A link's own terms in the adjoint, in world axes about its origin: its
// Newton-Euler wrench (moment n, force f; h = R m c)
//   f = m A + al x h + w x (w x h),  n = Io al + w x (Io w) + h x A
// and the gradients of wb . n + ub . f with respect to w, al and A,
//   gA = m ub + wb x h,  gal = Io wb + h x ub,
//   gw = (Io w) x wb + Io (wb x w) + grad_w [ub . (w x (w x h))],
// in o[15] = n, f, gw, gal, gA.  Four products with Io: it is rotated to the
// world once (45 operations, against 54 to rotate their arguments in and
// results out).
__device__ __forceinline__ void link_adjoint(const float* R, const float* I, const float* w,
                                             const float* al, const float* A, const float* wb,
                                             const float* ub, float* o) {
  float T[9], J[10], h[3];
#pragma unroll
  for (int i = 0; i < 3; ++i) rot_inertia(I, R + 3 * i, T + 3 * i);  // rows of R Io
  J[0] = I[0];
  J[4] = dot3(T, R);
  J[5] = dot3(T + 3, R + 3);
  J[6] = dot3(T + 6, R + 6);
  J[7] = dot3(T, R + 3);
  J[8] = dot3(T, R + 6);
  J[9] = dot3(T + 3, R + 6);
  rot(R, I + 1, h);
  float Iw[3], c[3];
  rot_inertia(J, w, Iw);
  rot_inertia(J, al, o);
  cross3_acc(w, Iw, o);
  cross3_acc(h, A, o);  // n
#pragma unroll
  for (int i = 0; i < 3; ++i) o[3 + i] = J[0] * A[i];
  cross3_acc(al, h, o + 3);
  centripetal_acc<1>(w, h, o + 3);  // f
  cross3(wb, w, c);
  rot_inertia(J, c, o + 6);
  cross3_acc(Iw, wb, o + 6);
  centripetal_grad(w, h, ub, o + 6);  // gw
  rot_inertia(J, wb, o + 9);
  cross3_acc(h, ub, o + 9);  // gal
#pragma unroll
  for (int i = 0; i < 3; ++i) o[12 + i] = J[0] * ub[i];
  cross3_acc(wb, h, o + 12);  // gA
}

// A thread's slot in shared memory for the upstream gradient rows that the
// next close reads: 6 float4 at p[q * stride], the link's pose gradient row
// (12 floats), then its first run of 4 sphere gradients.  Asynchronous copies
// (cp.async, bypassing L1) fill it while the sweep computes the link's push
// (a leaf) or its child's close, and the close waits for them: the rows' global
// latency no longer sits on the close's critical path.
struct GradSlot {
  float4* p = nullptr;
  int stride = 0;
};
constexpr int kGradSlotBytes = 6 * 16;  // a thread's slot
// the slots of a block behind `after` (any float address in dynamic shared
// memory), rounded up to 16 bytes; the block reserves kGradSlotBytes a thread
// plus 16 bytes for the rounding
__device__ __forceinline__ GradSlot grad_slot_of(float* after) {
  const uintptr_t a = reinterpret_cast<uintptr_t>(after);
  GradSlot g;
  g.p = reinterpret_cast<float4*>(after + ((16 - (a & 15)) & 15) / 4) + threadIdx.x;
  g.stride = blockDim.x;
  return g;
}
__device__ __forceinline__ void cp16(float4* dst, const void* src) {
  const unsigned a = static_cast<unsigned>(__cvta_generic_to_shared(dst));
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(a), "l"(src));
}

// With a fused cost (FC, fc) the sweep computes g_tau = [tau > hi] -
// [tau < lo] + 2 e qd^2 tau and g_dmin = -w [d_min < 0] itself, adds the
// cost's direct qd / qdd gradients (2 length qd + 2 e qd tau^2, 2 smooth qdd)
// to the outputs of the joint's link, and returns the cost terms of the joints
// of the links it owns (the caller adds the collision term and the segments'
// shares).  Needs one link per joint (no shared mimic joints).
// FC: compiled with the fused cost (a separate instantiation, so that the
// plain sweep keeps its register allocation).  gs: the thread's gradient-row
// slot, or none (the rows are then read with plain loads at each close).
template <bool FC, class St>
__device__ __forceinline__ float tree_bwd_seg(const DevRobot& r, const BwdArgs& A,
                                              const FusedCost& fc, const St& st, int64_t b,
                                              const Seg& sg, GradSlot gs = GradSlot{}) {
  const int64_t B = A.B;
  float cost_part = 0.0f;
  const int n = r.n;
  BEnt stk[TMAXD];
  if (r.mimic_shared)
    for (int j = 0; j < r.d; ++j) {
      A.gq[(int64_t)j * B + b] = 0.0f;
      A.gqd[(int64_t)j * B + b] = 0.0f;
      A.gqdd[(int64_t)j * B + b] = 0.0f;
    }
  // the worst pair's gradient: u = g_dmin (c_i - c_j) / |c_i - c_j|, needed
  // only by the segment that owns one of the pair's links
  auto owned = [&](int k) {
    if (!sg.slot) return true;
    const int p = __ldg(r.dfs_pos + k);
    return p >= sg.p0 && p < sg.p1;
  };
  int pl1 = -1, pl2 = -1, ps1 = 0, ps2 = 0;
  float u[3] = {0.0f, 0.0f, 0.0f};
  if (A.g_dmin || (FC && fc.d_min)) {
    const int wp = A.worst[b];
    const float gd = FC ? (__ldg(fc.d_min + b) < 0.0f ? -fc.w : 0.0f) : A.g_dmin[b];
    if (wp >= 0 && wp < r.P && gd != 0.0f) {
      const int2 ij = __ldg(r.pairs + wp);
      const int l1 = __ldg(r.sph_link + ij.x), l2 = __ldg(r.sph_link + ij.y);
      if (owned(l1) || owned(l2)) {
        ps1 = ij.x;
        ps2 = ij.y;
        pl1 = l1;
        pl2 = l2;
        float dx, dy, dz;
        if (A.wdiff) {  // from the pair stage: the same arithmetic on the same poses
          dx = __ldg(A.wdiff + 3 * b);
          dy = __ldg(A.wdiff + 3 * b + 1);
          dz = __ldg(A.wdiff + 3 * b + 2);
        } else {  // place the two spheres from their links' ancestor chains
          float P1[12], P2[12], c1[3], c2[3];
          chain_pose(r, pl1, st, P1);
          chain_pose(r, pl2, st, P2);
          const float4 s1 = __ldg(r.sph + ps1), s2 = __ldg(r.sph + ps2);
          const float q1[3] = {s1.x, s1.y, s1.z}, q2[3] = {s2.x, s2.y, s2.z};
          rot(P1, q1, c1);
          rot(P2, q2, c2);
          dx = (c1[0] + P1[9]) - (c2[0] + P2[9]);
          dy = (c1[1] + P1[10]) - (c2[1] + P2[10]);
          dz = (c1[2] + P1[11]) - (c2[2] + P2[11]);
        }
        const float nrm = sqrtf(fmaf(dz, dz, fmaf(dy, dy, dx * dx)));
        const float sc = nrm > 0.0f ? gd / nrm : 0.0f;
        u[0] = dx * sc;
        u[1] = dy * sc;
        u[2] = dz * sc;
      }
    }
  }

  // The state in registers: the pre-order data (W, w, al, A, wb, ub) of the
  // last pushed link after a push, of the closed link's parent after a close;
  // the just-pushed link's torque adjoint (ctb, valid while fresh); and the
  // accumulated children's sums of the entry the post-order closes next (an
  // unwinding chain passes them on in registers; they are stored when a push
  // interrupts).
  float cW[12], cw[3], cal[3], cA[3], cwb[3], cub[3], ctb = 0.0f;
  bool fresh = false;
  float ps[kSums];
  int pdep = -1;
  // bit e: entry e is an ancestor replayed for this segment (no own terms),
  // its acc holds children's sums
  uint32_t replayed = 0u, accv = 0u;
  int lcs = 0;  // where the last pushed link's ancestor chain starts (the stack holds it)
  const bool kin_grad = A.g_pose != nullptr || A.g_sph != nullptr;
  // sphere gradients of a link as float4 triples: the robot's spheres come
  // in runs of 4 (then b S + s is a multiple of 4) and the array (a slice of
  // a packed batch, possibly) is 16-byte aligned
  const bool sph4 = A.g_sph != nullptr && r.sph_vec4 &&
                    (reinterpret_cast<uintptr_t>(A.g_sph) & 15u) == 0;
  // the link whose gradient rows are on their way into the slot (-1: none)
  int pend = -1;
  const bool use_slot = gs.p != nullptr && kin_grad;
  auto issue = [&](int k) {
    if (A.g_pose) {
      const float4* g4 = reinterpret_cast<const float4*>(A.g_pose + (b * n + k) * 12);
      cp16(gs.p, g4);
      cp16(gs.p + gs.stride, g4 + 1);
      cp16(gs.p + 2 * gs.stride, g4 + 2);
    }
    if (sph4) {
      const int e0 = __ldg(r.ls_start + k);
      if (__ldg(r.ls_start + k + 1) > e0) {
        const float4* g4 = reinterpret_cast<const float4*>(A.g_sph + (b * r.S + __ldg(r.ls_sph + e0)) * 3);
        cp16(gs.p + 3 * gs.stride, g4);
        cp16(gs.p + 4 * gs.stride, g4 + 1);
        cp16(gs.p + 5 * gs.stride, g4 + 2);
      }
    }
    asm volatile("cp.async.commit_group;");
    pend = k;
  };

  // gradient wrench of link k's kinematic outputs (pose, spheres, the worst
  // pair's spheres) in world axes about its origin: the points' gradients
  // join the rotation gradient G, whose wrench is the sum of the crosses of
  // R's columns with G's
  auto wrench = [&](int k, float* w) {
    float G[9];
#pragma unroll
    for (int i = 0; i < 9; ++i) G[i] = 0.0f;
    float* f = w + 3;
    f[0] = f[1] = f[2] = 0.0f;
    const bool slot = pend == k;
    if (slot) asm volatile("cp.async.wait_group 0;" ::: "memory");
    pend = -1;
    if (A.g_pose) {
      const float4* g4 = reinterpret_cast<const float4*>(A.g_pose + (b * n + k) * 12);
      const float4 x0 = slot ? gs.p[0] : __ldg(g4), x1 = slot ? gs.p[gs.stride] : __ldg(g4 + 1),
                   x2 = slot ? gs.p[2 * gs.stride] : __ldg(g4 + 2);
      G[0] = x0.x; G[1] = x0.y; G[2] = x0.z; G[3] = x0.w; G[4] = x1.x;
      G[5] = x1.y; G[6] = x1.z; G[7] = x1.w; G[8] = x2.x;
      f[0] = x2.y; f[1] = x2.z; f[2] = x2.w;
    }
    if (sph4) {  // runs of 4 spheres: three float4 loads a run
      const int e1 = __ldg(r.ls_start + k + 1);
      const int ef = __ldg(r.ls_start + k);
      for (int e = ef; e < e1; e += 4) {
        const int s = __ldg(r.ls_sph + e);
        const float4* g4 = reinterpret_cast<const float4*>(A.g_sph + (b * r.S + s) * 3);
        const bool fs = slot && e == ef;
        const float4 x0 = fs ? gs.p[3 * gs.stride] : __ldg(g4),
                     x1 = fs ? gs.p[4 * gs.stride] : __ldg(g4 + 1),
                     x2 = fs ? gs.p[5 * gs.stride] : __ldg(g4 + 2);
        const float gg[12] = {x0.x, x0.y, x0.z, x0.w, x1.x, x1.y, x1.z, x1.w, x2.x, x2.y, x2.z, x2.w};
#pragma unroll
        for (int i = 0; i < 4; ++i) point_grad(__ldg(r.sph + s + i), gg + 3 * i, G, f);
      }
    } else if (A.g_sph) {
      const int e1 = __ldg(r.ls_start + k + 1);
      for (int e = __ldg(r.ls_start + k); e < e1; ++e) {
        const int s = __ldg(r.ls_sph + e);
        const float* g = A.g_sph + (b * r.S + s) * 3;
        const float gg[3] = {__ldg(g), __ldg(g + 1), __ldg(g + 2)};
        point_grad(__ldg(r.sph + s), gg, G, f);
      }
    }
    if (k == pl1) point_grad(__ldg(r.sph + ps1), u, G, f);
    if (k == pl2) {
      const float mu[3] = {-u[0], -u[1], -u[2]};
      point_grad(__ldg(r.sph + ps2), mu, G, f);
    }
    const float* R = cW;
    w[0] = w[1] = w[2] = 0.0f;
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      const float rc[3] = {R[j], R[3 + j], R[6 + j]}, gc[3] = {G[j], G[3 + j], G[6 + j]};
      cross3_acc(rc, gc, w);
    }
  };

  // post-order of the link at depth e; the registers hold its state; tgt:
  // the closes go on down to depth tgt
  auto close = [&](int e, int tgt) {
    // the link at depth e with its joint, type and rotation flag, one load
    const int cm = __ldg(r.chain_m + lcs + e);
    const int k = cm & 0xFF;
    const bool own = !((replayed >> e) & 1u);
    // own terms (link_adjoint, minus the external wrench) and the gradient
    // wrench of the kinematic outputs
    float o[kSums];
    if (own) {
      float I[10];
      load_inertia(r, k, I);
      link_adjoint(cW, I, cw, cal, cA, cwb, cub, o);
      if (A.fext) {
        const float* fe = A.fext + (b * n + k) * 6;
        const float xn[3] = {__ldg(fe), __ldg(fe + 1), __ldg(fe + 2)};
        const float xf[3] = {__ldg(fe + 3), __ldg(fe + 4), __ldg(fe + 5)};
        float t[3];
        rot(cW, xn, t);
#pragma unroll
        for (int i = 0; i < 3; ++i) o[i] -= t[i];
        rot(cW, xf, t);
#pragma unroll
        for (int i = 0; i < 3; ++i) o[3 + i] -= t[i];
      }
      if (kin_grad || k == pl1 || k == pl2) {
        wrench(k, o + 15);
        // the next close's rows, while this one computes
        if (use_slot && e - 1 >= tgt && !((replayed >> (e - 1)) & 1u))
          issue(__ldg(r.chain_m + lcs + e - 1) & 0xFF);
      } else {
#pragma unroll
        for (int i = 15; i < kSums; ++i) o[i] = 0.0f;
      }
    } else {
#pragma unroll
      for (int i = 0; i < kSums; ++i) o[i] = 0.0f;
    }
    // plus the children's sums
    if (pdep == e) {
#pragma unroll
      for (int i = 0; i < kSums; ++i) o[i] += ps[i];
    } else if ((accv >> e) & 1u) {
      const BEnt& E = stk[e];
#pragma unroll
      for (int i = 0; i < kSums; ++i) o[i] += E.acc[i];
    }
    pdep = -1;
    float *sn = o, *sf = o + 3, *gw = o + 6, *gal = o + 9, *gA = o + 12, *Wn = o + 15,
          *Wf = o + 18;
    const int j = ((cm >> 8) & 0x1FF) - 1;
    const int jt = (cm >> 17) & 3;
    const float4 a4 = ldp(reinterpret_cast<const float4*>(r.axis) + k);
    const float ax[3] = {a4.x, a4.y, a4.z};
    const float mm = ldp(reinterpret_cast<const float2*>(r.mimic) + k).x;
    const float vq = j >= 0 ? mm * st.vel(j) : 0.0f;
    const float aq = j >= 0 ? mm * st.acc(j) : 0.0f;
    const float tb = fresh ? ctb : (e > 0 ? stk[e].tb : 0.0f);
    float s[3];
    rot(cW, ax, s);
    // The joint's gradients.  Turning a revolute joint turns everything the
    // subtree holds; what enters it from the parent stays, so with the sums
    // as the gradients of the link's own w, al, A, wb, ub
    //   gq   = s . [Wn - w x gw - al x gal - A x gA - wb x n - ub x f],
    //   gqd  = s . gw + (w x s) . gal,  gqdd = s . gal,
    // and w_pa also moves al through w_pa x s qd: gw += qd s x gal.  Sliding
    // a prismatic joint moves the subtree's origin along s (through r).
    float gq = 0.0f, gqd = 0.0f, gqdd = 0.0f;
    if (jt == 1) {
      float t[3] = {Wn[0], Wn[1], Wn[2]}, c[3];
      cross3_sub(cw, gw, t);
      cross3_sub(cal, gal, t);
      cross3_sub(cA, gA, t);
      cross3_sub(cwb, sn, t);
      cross3_sub(cub, sf, t);
      gq = dot3(s, t);
      cross3(cw, s, c);
      gqd = dot3(s, gw) + dot3(c, gal);
      gqdd = dot3(s, gal);
      const float sq[3] = {s[0] * vq, s[1] * vq, s[2] * vq};
      cross3_acc(sq, gal, gw);
      // the parent's w, al, wb
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        cw[i] -= sq[i];
        cal[i] = fmaf(-s[i], aq, fmaf(-vq, c[i], cal[i]));
        cwb[i] = fmaf(-s[i], tb, cwb[i]);
      }
    } else if (jt == 2) {
      float t[3] = {Wf[0], Wf[1], Wf[2]}, c[3], c2[3];
      // gA . (al x s + w x (w x s)) + f . (wb x s) + s . Wf
      cross3_acc(gA, cal, t);
      cross3_acc(sf, cwb, t);
      cross3(cw, s, c);
      cross3(cw, c, c2);
      gq = dot3(s, t) + dot3(gA, c2);
      gqd = 2.0f * dot3(c, gA);
      gqdd = dot3(s, gA);
      const float sq[3] = {2.0f * vq * s[0], 2.0f * vq * s[1], 2.0f * vq * s[2]};
      cross3_acc(sq, gA, gw);
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        cA[i] = fmaf(-s[i], aq, fmaf(-2.0f * vq, c[i], cA[i]));
        cub[i] = fmaf(-s[i], tb, cub[i]);
      }
    }
    if (FC && j >= 0) {
      float dqd = 0.0f, dqdd = 0.0f;  // the cost's direct gradients, once per joint
      if (own) {
        const int64_t at = (int64_t)j * B + b;
        const float tj = __ldg(fc.tau + at), vj = st.vel(j), aj = st.acc(j);
        dqd = 2.0f * (fc.length * vj + fc.e * (vj * tj) * tj);
        dqdd = 2.0f * fc.smooth * aj;
      }
      float* p0 = seg_part(sg, k, 0);
      if (p0) {
        const size_t o = (size_t)sg.ns * sg.G * 32;
        p0[0] = mm * gq;
        p0[o] = mm * gqd + dqd;
        p0[2 * o] = mm * gqdd + dqdd;
      } else {
        A.gq[(int64_t)j * B + b] = mm * gq;
        A.gqd[(int64_t)j * B + b] = mm * gqd + dqd;
        A.gqdd[(int64_t)j * B + b] = mm * gqdd + dqdd;
      }
    } else if (j >= 0) {
      float* p0 = seg_part(sg, k, 0);
      if (p0) {
        const size_t o = (size_t)sg.ns * sg.G * 32;
        p0[0] = mm * gq;
        p0[o] = mm * gqd;
        p0[2 * o] = mm * gqdd;
      } else {
        float* o0 = A.gq + (int64_t)j * B + b;
        float* o1 = A.gqd + (int64_t)j * B + b;
        float* o2 = A.gqdd + (int64_t)j * B + b;
        if (r.mimic_shared) {
          *o0 += mm * gq;
          *o1 += mm * gqd;
          *o2 += mm * gqdd;
        } else {
          *o0 = mm * gq;
          *o1 = mm * gqd;
          *o2 = mm * gqdd;
        }
      }
    }
    fresh = false;
    if (e > 0) {
      float rv[3];  // the offset from the parent's origin
      float L[12], Wp[12];
      const float th = j >= 0 ? joint_var(r, k, st.pos(j)) : 0.0f;
      local_xf_m<true>(r, k, th, jt, ((cm >> 19) & 1) != 0, L, L + 9);
      uncompose(cW, L, Wp, rv);
#pragma unroll
      for (int i = 0; i < 12; ++i) cW[i] = Wp[i];
      cross3_sub(cal, rv, cA);
      centripetal_acc<-1>(cw, rv, cA);
      cross3_sub(cwb, rv, cub);
      // the sums about the parent's origin
      centripetal_grad(cw, rv, gA, gw);
      cross3_acc(rv, gA, gal);
      cross3_acc(rv, sf, sn);
      cross3_acc(rv, Wf, Wn);
      const BEnt& P = stk[e - 1];
      const bool has = (accv >> (e - 1)) & 1u;
      accv &= ~(1u << (e - 1));  // taken over by the pending registers
#pragma unroll
      for (int i = 0; i < kSums; ++i) ps[i] = has ? P.acc[i] + o[i] : o[i];
      pdep = e - 1;
    }
  };
  auto flush = [&]() {  // the pending children's sums go to their entry
    if (pdep >= 0) {
      BEnt& P = stk[pdep];
#pragma unroll
      for (int i = 0; i < kSums; ++i) P.acc[i] = ps[i];
      accv |= 1u << pdep;
      pdep = -1;
    }
  };

  // pre-order of link k at depth dep (the registers hold its parent's state);
  // own = false replays an ancestor of the segment (its own contributions
  // are zero)
  auto push = [&](int k, int dep, bool own, int ky, int cs) {
    const int j = (ky & 0xFFFF) - 1, nch = (ky >> 16) & 0xFF, jt = (ky >> 24) & 3;
    float L[12];
    {
      const float th = j >= 0 ? joint_var(r, k, st.pos(j)) : 0.0f;
      local_xf_m<true>(r, k, th, jt, ((ky >> 26) & 1) != 0, L, L + 9);
    }
    const float4 a4 = ldp(reinterpret_cast<const float4*>(r.axis) + k);
    const float ax[3] = {a4.x, a4.y, a4.z};
    const float mm = ldp(reinterpret_cast<const float2*>(r.mimic) + k).x;
    const float vq = j >= 0 ? mm * st.vel(j) : 0.0f;
    const float aq = j >= 0 ? mm * st.acc(j) : 0.0f;
    // the adjoint of the force sweep's torque term: taubar of the joint
    float tb = 0.0f;
    if (FC && j >= 0) {  // the cost's torque gradient, as the cost kernel forms it
      const float t = __ldg(fc.tau + (int64_t)j * B + b), l = __ldg(fc.lo + j),
                  h = __ldg(fc.hi + j);
      const float v = st.vel(j), a = st.acc(j);
      const float vt = v * t;
      float gt = 2.0f * fc.e * v * vt;
      gt += (t > h ? 1.0f : 0.0f) - (t < l ? 1.0f : 0.0f);
      tb = mm * gt;
      if (own) {
        float c = fmaf(fc.smooth * a, a, 0.0f);
        c = fmaf(fc.length * v, v, c);
        c = fmaf(fc.e * vt, vt, c);
        c += fmaxf(0.0f, t - h) + fmaxf(0.0f, l - t);
        cost_part += c;
      }
    } else if (!FC && j >= 0 && A.g_tau) {
      tb = mm * __ldg(A.g_tau + (int64_t)j * B + b);
    }
    // the link's state: pose, motion, and the torques' virtual motion
    // wb = wb_pa + s tb, ub = ub_pa + wb_pa x r (prismatic: ub + s tb)
    float Wn[12], s[3], rv[3], wn[3], aln[3], An[3];
    if (dep > 0) {
      compose(cW, L, Wn, rv);
      rot(Wn, ax, s);
      joint_motion(jt, s, rv, vq, aq, cw, cal, cA, wn, aln, An);
      cross3_acc(cwb, rv, cub);
    } else {
#pragma unroll
      for (int i = 0; i < 12; ++i) Wn[i] = L[i];
      rot(Wn, ax, s);
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        cw[i] = cal[i] = cwb[i] = cub[i] = rv[i] = 0.0f;
        cA[i] = r.abase[i];
      }
      joint_motion(jt, s, rv, vq, aq, cw, cal, cA, wn, aln, An);
    }
#pragma unroll
    for (int i = 0; i < 12; ++i) cW[i] = Wn[i];
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      cw[i] = wn[i];
      cal[i] = aln[i];
      cA[i] = An[i];
      if (jt == 2)
        cub[i] = fmaf(s[i], tb, cub[i]);
      else
        cwb[i] = fmaf(s[i], tb, cwb[i]);
    }
    ctb = tb;
    fresh = true;
    lcs = cs;
    const uint32_t bit = 1u << dep;
    accv &= ~bit;
    replayed = own ? (replayed & ~bit) : (replayed | bit);
    if (nch > 0) stk[dep].tb = tb;
    if (own && A.g_fext) {  // dL/df_ext,k = -(wb, ub) in link coordinates
      float* o = A.g_fext + (b * n + k) * 6;
      float t[6];
      rotT(cW, cwb, t);
      rotT(cW, cub, t + 3);
#pragma unroll
      for (int i = 0; i < 6; ++i) o[i] = -t[i];
    }
  };

  int sp = 0;
  if (sg.p0 > 0) {  // replay the proper ancestors of the first link
    const int k0 = __ldg(r.dfs + sg.p0).x;
    const int c0 = __ldg(r.chain_start + k0), c1 = __ldg(r.chain_start + k0 + 1);
    for (int c = c0; c < c1 - 1; ++c) {
      const int a = __ldg(r.chain + c);
      push(a, c - c0, false, packed_link(r, a), __ldg(r.chain_start + a));
    }
    sp = c1 - 1 - c0;
  }
  for (int pos = sg.p0; pos < sg.p1; ++pos) {
    const int2 kd = __ldg(r.dfs_kj + pos);  // link | depth << 8 | chain start << 16, joint word
    const int k = kd.x & 0xFF, dep = (kd.x >> 8) & 0xFF;
    const int2 kn = pos + 1 < sg.p1 ? __ldg(r.dfs_kj + pos + 1) : make_int2(0, 0);
    // L2 prefetch of the next link's joint inputs.  The gradient rows its
    // close reads are not prefetched: measured slower (the humanoid's
    // backward 0.218 -> 0.210 ms without)
    if (pos + 1 < sg.p1) {
      const int jn = (kn.y & 0xFFFF) - 1;
      if (jn >= 0) {
        st.prefetch(jn, true);
        if (A.g_tau) pf(A.g_tau + (int64_t)jn * B + b);
        if (FC) pf(fc.tau + (int64_t)jn * B + b);
      }
    }
    while (sp > dep) close(--sp, dep);
    flush();
    sp = dep + 1;
    // a link closed right after its push (a leaf, or the segment's last
    // link): its rows start on their way now
    if (use_slot && (pos + 1 >= sg.p1 || ((kn.x >> 8) & 0xFF) <= dep)) issue(k);
    push(k, dep, true, kd.y, kd.x >> 16);
  }
  while (sp > 0) close(--sp, 0);
  flush();
  if (pend >= 0) asm volatile("cp.async.wait_group 0;" ::: "memory");
  return cost_part;
}

// the whole sweep of one configuration; with a fused cost it also writes the
// configuration's cost (joint terms, then the collision term)
__device__ __forceinline__ void tree_bwd_one(const DevRobot& r, const BwdArgs& A, int64_t b) {
  tree_bwd_seg<false>(r, A, FusedCost{}, ArrayStates{A.q, A.qd, A.qdd, A.B, b}, b,
                      whole_sweep(r));
}

template <class St>
__device__ __forceinline__ void tree_bwd_cost_one(const DevRobot& r, const BwdArgs& A,
                                                  const FusedCost& fc, const St& st, int64_t b) {
  const float c = tree_bwd_seg<true>(r, A, fc, st, b, whole_sweep(r));
  if (fc.cost) fc.cost[b] = fc.d_min ? fmaf(fc.w, fmaxf(0.0f, -__ldg(fc.d_min + b)), c) : c;
}

}  // namespace wbe
