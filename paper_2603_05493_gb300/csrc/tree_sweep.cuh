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
// unit circle (UNIT in local_xf_q): gradient error against 64 bits 3.5e-6 ->
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

// The walk: one word a DFS position with what steers the sweep at it --
// depth, joint and its type, the parent's position.  The single-robot kernels
// take the words as a kernel argument: read at a warp-uniform position they
// come from the constant bank into uniform registers, so the sweep's branches
// need no reconvergence (with the words in global memory a fifth of the
// forward's instructions were branches, barriers and moves around them).
__device__ __forceinline__ int wk_dep(uint32_t w) { return w & 31; }
__device__ __forceinline__ bool wk_branch(uint32_t w) { return (w >> 5) & 1; }  // >= 2 children
__device__ __forceinline__ int wk_jt(uint32_t w) { return (w >> 6) & 3; }
__device__ __forceinline__ bool wk_ident(uint32_t w) { return (w >> 8) & 1; }
__device__ __forceinline__ bool wk_leaf(uint32_t w) { return (w >> 9) & 1; }
__device__ __forceinline__ int wk_j(uint32_t w) { return (w >> 10) & 255; }
__device__ __forceinline__ int wk_par(uint32_t w) { return (w >> 18) & 255; }

// TABLE: the ancestors that a segment replays come from a table.  The backward climbs
// to each of them from the segment's first link instead: with the table's address
// beside its state it spilled (128 registers).
template <bool TABLE>
struct ConstWalk {
  static constexpr bool kSpheres = true;  // the spheres are staged behind the records
  const WalkTab& t;
  __device__ __forceinline__ uint32_t operator()(int pos) const { return t.w[pos]; }
  // the position of the ancestor at depth c of p0, the first link of segment g of G
  __device__ __forceinline__ int ancestor(int p0, int G, int g, int c) const {
    if (TABLE) return t.rep[G + g][c];
    int pos = p0;
    for (uint32_t w = t.w[pos]; wk_dep(w) > c; w = t.w[pos]) pos = wk_par(w);
    return pos;
  }
};
struct SharedWalk {  // the batch's: staged with the link records, made uniform by a shuffle
  static constexpr bool kSpheres = false;
  const uint32_t* w;    // the walk words
  const uint32_t* rep;  // [kRepDepth] the ancestors of the second of two segments' first link
  __device__ __forceinline__ uint32_t operator()(int pos) const {
    return __shfl_sync(0xffffffffu, w[pos], 0);
  }
  __device__ __forceinline__ int ancestor(int, int, int g, int c) const {
    return g == 0 ? 0 : (int)__shfl_sync(0xffffffffu, rep[c], 0);
  }
};

// One segment of a segmented sweep (see above).  part == nullptr: the whole
// DFS order, outputs written directly.
struct Seg {
  int p0, p1;   // DFS positions this segment owns
  int g, G;     // segment index, segments per configuration
  float* part;  // partial outputs of this group: [nout][ns][G][32]
  int ns;       // shared slots
  int lane;
  // forward sweep with its force stack in shared memory: this thread's
  // entry 0, and the stride of the [depth][3][threads] layout (the block's
  // threads)
  float2* fst = nullptr;
  int fstr = 0;
};

__device__ __forceinline__ Seg whole_sweep(const DevRobot& r) {
  return Seg{0, r.n, 0, 1, nullptr, 0, 0};
}

// the robot's spheres, behind its staged records (the backward reads a link's
// at its close: humanoid48 0.290 -> 0.272 ms at 99999 configurations)
__device__ __forceinline__ void stage_spheres(const DevRobot& r, float4* rec) {
  for (int i = threadIdx.x; i < r.S; i += blockDim.x) rec[8 * r.n + i] = __ldg(r.sph + i);
}

// Copies the robot's link records into shared memory (kRecWords floats a
// link, in DFS order; see DevRobot::recs) with the inertias and the shared
// output slots of segment plan t (t < 0: none); thread i of nt.
__device__ __forceinline__ void stage_recs(const DevRobot& r, int t, float4* dst, int i0, int nt) {
  for (int i = i0; i < 8 * r.n; i += nt) {
    float4 v = __ldg(r.recs + i);
    const int w = i & 7;
    if (w >= 4) {
      const int k = __ldg(r.dfs + (i >> 3)).x;
      const float* in = r.inert + 10 * k;
      if (w < 6) {
        const float* x = in + 4 * (w - 4);
        v = make_float4(__ldg(x), __ldg(x + 1), __ldg(x + 2), __ldg(x + 3));
      } else if (w == 6) {
        v.x = __ldg(in + 8);
        v.y = __ldg(in + 9);
      } else {
        v.y = __int_as_float(t >= 0 ? (int)__ldg(r.seg_slot + t * r.n + k) : -1);
      }
    }
    dst[i] = v;
  }
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

// where the partial output o of the link with record q goes, or nullptr for a
// direct write
__device__ __forceinline__ float* seg_part(const Seg& sg, const float4* q, int o) {
  if (!sg.part) return nullptr;
  const int s = __float_as_int(q[7].y);
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

// y += Io x for the rotational part of the compact inertia
__device__ __forceinline__ void rot_inertia_acc(const float* I, const float* x, float* y) {
  y[0] = fmaf(I[8], x[2], fmaf(I[7], x[1], fmaf(I[4], x[0], y[0])));
  y[1] = fmaf(I[9], x[2], fmaf(I[5], x[1], fmaf(I[7], x[0], y[1])));
  y[2] = fmaf(I[6], x[2], fmaf(I[9], x[1], fmaf(I[8], x[0], y[2])));
}
// y = Io x
__device__ __forceinline__ void rot_inertia(const float* I, const float* x, float* y) {
  y[0] = fmaf(I[8], x[2], fmaf(I[7], x[1], I[4] * x[0]));
  y[1] = fmaf(I[9], x[2], fmaf(I[5], x[1], I[7] * x[0]));
  y[2] = fmaf(I[6], x[2], fmaf(I[9], x[1], I[8] * x[0]));
}

// world pose W <- W o L (12 floats each); t: the offset of the new origin
// from the old one
__device__ __forceinline__ void compose(float* W, const float* L, float* t) {
  rot(W, L + 9, t);
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    const float a = W[3 * i], b = W[3 * i + 1], c = W[3 * i + 2];
#pragma unroll
    for (int j = 0; j < 3; ++j)
      W[3 * i + j] = fmaf(c, L[6 + j], fmaf(b, L[3 + j], a * L[j]));
    W[9 + i] += t[i];
  }
}

// local transform of the link with record q for its joint's value qj
template <bool UNIT = false>
__device__ __forceinline__ void link_local(const float4* q, uint32_t w, float qj, float* L) {
  const int jt = wk_jt(w);
  const float th = jt ? fmaf(q[3].w, qj, q[6].z) : 0.0f;
  local_xf_q<UNIT>(q, q[3], th, jt, wk_ident(w), L, L + 9);
}

__device__ __forceinline__ void rec_inertia(const float4* q, float* I) {
  const float4 a = q[4], b = q[5], c = q[6];
  I[0] = a.x; I[1] = a.y; I[2] = a.z; I[3] = a.w;
  I[4] = b.x; I[5] = b.y; I[6] = b.z; I[7] = b.w;
  I[8] = c.x; I[9] = c.y;
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

// MODE kFwdPose: poses only (its own instantiation: without the dynamics'
// registers the poses-only sweep of the humanoid takes half the registers);
// kFwdLocal: torques too when A.tau is given; kFwdShared: with torques, the
// accumulated forces F of the stack in shared memory (sg.fst) instead of the
// thread's local stack.  All 32 lanes of the warp take part; a
// lane past the end sweeps the last configuration again and writes the same
// values (act = false keeps it out of read-modify-write outputs).
enum FwdMode { kFwdPose, kFwdLocal, kFwdShared };
template <int MODE, class WK, class St>
__device__ __forceinline__ void tree_fwd_seg(const DevRobot& r, const float4* rec, const WK& wk,
                                             const FwdArgs& A, const St& st, int64_t b, bool act,
                                             const Seg& sg) {
  constexpr bool FS = MODE == kFwdShared;
  const int64_t B = A.B;
  const bool dyn = FS || (MODE != kFwdPose && A.tau != nullptr);
  FEnt stk[TMAXD];
  if (dyn && r.mimic_shared && act)
    for (int j = 0; j < r.d; ++j) A.tau[(int64_t)j * B + b] = 0.0f;
  float* const pose_b = A.pose ? A.pose + b * r.n * 12 : nullptr;
  // Register copies that spare most stack loads: the pre-order data of the
  // last pushed entry (never changes while the entry is on the stack; a link
  // pushed right after its parent finds it here), and the accumulated force
  // of the entry that the post-order closes next (an unwinding chain passes
  // it on in registers; it is stored when a push interrupts).
  float cW[12], cv[6], ca[6], pF[6];
#pragma unroll
  for (int i = 0; i < 6; ++i) cv[i] = ca[i] = pF[i] = 0.0f;
#pragma unroll
  for (int i = 0; i < 12; ++i) cW[i] = 0.0f;
  int cdep = -1, pdep = -1;
  int ckp = 0;  // the position the next close takes: the last pushed one, then parents
  // its joint's value: the push's, then loaded a close ahead (a load at the
  // head of every close sat on its critical path: humanoid48 0.066 -> 0.060
  // ms; the backward, whose closes use it after the own terms, gains nothing)
  float kq = 0.0f;

  auto load_F = [&](int e, float* F) {
    if (FS) {
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        const float2 x = sg.fst[(3 * e + i) * sg.fstr];
        F[2 * i] = x.x;
        F[2 * i + 1] = x.y;
      }
    } else {
#pragma unroll
      for (int i = 0; i < 6; ++i) F[i] = stk[e].F[i];
    }
  };
  auto close = [&](int e) {
    const uint32_t w = wk(ckp);
    const float4* q = rec + 8 * ckp;
    ckp = wk_par(w);
    const int j = wk_j(w), jt = wk_jt(w);
    const float qj = kq;
    if (e > 0) {
      const uint32_t wp = wk(ckp);
      kq = wk_jt(wp) ? st.pos(wk_j(wp)) : 0.0f;
    }
    if (pdep != e) load_F(e, pF);
    pdep = -1;
    if (jt) {
      const float4 a4 = q[3];
      const float ax[3] = {a4.x, a4.y, a4.z};
      const float t = a4.w * (jt == 1 ? dot3(ax, pF) : dot3(ax, pF + 3));
      float* pt = seg_part(sg, q, 0);
      if (pt) {
        *pt = t;
      } else {
        float* dst = A.tau + (int64_t)j * B + b;
        if (!r.mimic_shared)
          *dst = t;
        else if (act)
          *dst += t;
      }
    }
    if (e > 0) {
      float L[12], up[6], F[6];
      load_F(e - 1, F);
      link_local(q, w, qj, L);
      xf_force_T(L, L + 9, pF, up);
#pragma unroll
      for (int i = 0; i < 6; ++i) pF[i] = F[i] + up[i];
      pdep = e - 1;
    }
  };
  auto flush = [&]() {  // the pending force goes back to its stack entry
    if (pdep >= 0) {
      if (FS) {
#pragma unroll
        for (int i = 0; i < 3; ++i)
          sg.fst[(3 * pdep + i) * sg.fstr] = make_float2(pF[2 * i], pF[2 * i + 1]);
      } else {
#pragma unroll
        for (int i = 0; i < 6; ++i) stk[pdep].F[i] = pF[i];
      }
      pdep = -1;
    }
  };

  // pre-order of the link at pos; own = false replays an ancestor of the
  // segment (pose, v, a only; no output, no force of its own); pq, pqd, pqdd:
  // its joint's state
  auto push = [&](int pos, uint32_t w, bool own, float pq, float pqd, float pqdd) {
    const float4* q = rec + 8 * pos;
    const int dep = wk_dep(w), jt = wk_jt(w);
    FEnt& E = stk[dep];
    float L[12];
    link_local(q, w, pq, L);
    if (dep > 0) {
      if (dep != cdep + 1) {  // a later child: its parent's pre-order data from the stack
        const FEnt& P = stk[dep - 1];
#pragma unroll
        for (int i = 0; i < 12; ++i) cW[i] = P.W[i];
#pragma unroll
        for (int i = 0; i < 6; ++i) {
          cv[i] = P.v[i];
          ca[i] = P.a[i];
        }
      }
      float t[3];
      compose(cW, L, t);
    } else {
#pragma unroll
      for (int i = 0; i < 12; ++i) cW[i] = L[i];
#pragma unroll
      for (int i = 0; i < 6; ++i) cv[i] = ca[i] = 0.0f;
#pragma unroll
      for (int i = 0; i < 3; ++i) ca[3 + i] = r.abase[i];
    }
    cdep = dep;
    ckp = pos;
    kq = pq;
    if (wk_branch(w)) {
#pragma unroll
      for (int i = 0; i < 12; ++i) E.W[i] = cW[i];
    }
    const int k = __float_as_int(q[7].x) & 0xFF;
    if (own && pose_b) {
      float4* dst = reinterpret_cast<float4*>(pose_b + 12 * k);
      dst[0] = make_float4(cW[0], cW[1], cW[2], cW[3]);
      dst[1] = make_float4(cW[4], cW[5], cW[6], cW[7]);
      dst[2] = make_float4(cW[8], cW[9], cW[10], cW[11]);
    }
    if (dyn) {
      const float4 a4 = q[3];
      const float ax[3] = {a4.x, a4.y, a4.z};
      const float vq = a4.w * pqd, aq = a4.w * pqdd;
      float vn[6], an[6];
      rnea_va(L, L + 9, cv, ca, jt, ax, vq, aq, vn, an);
#pragma unroll
      for (int i = 0; i < 6; ++i) {
        cv[i] = vn[i];
        ca[i] = an[i];
      }
      // the force waits in the pending registers; a child's push stores it
      if (own) {
        float I[10];
        rec_inertia(q, I);
        rnea_force(I, cv, ca, pF);
        if (A.fext) {  // f_k = I a + v x* I v - f_ext,k
          const float* fe = A.fext + (b * r.n + k) * 6;
#pragma unroll
          for (int i = 0; i < 6; ++i) pF[i] -= __ldg(fe + i);
        }
      } else {
#pragma unroll
        for (int i = 0; i < 6; ++i) pF[i] = 0.0f;
      }
      if (wk_branch(w)) {
#pragma unroll
        for (int i = 0; i < 6; ++i) {
          E.v[i] = cv[i];
          E.a[i] = ca[i];
        }
      }
      pdep = dep;
    }
  };

  // One loop over the replayed proper ancestors of the first link and the
  // segment's links, one call site each for push and close; past the last
  // link everything closes.  The joint state of the link pushed next is
  // loaded one link ahead into registers, so that its latency overlaps the
  // current link's closes and push.
  const int nrep = wk_dep(wk(sg.p0)), total = nrep + sg.p1 - sg.p0;
  int sp = 0;
  int npos = wk.ancestor(sg.p0, sg.G, sg.g, 0);
  uint32_t nw = wk(npos);
  float nq = 0.0f, nqd = 0.0f, nqdd = 0.0f;
  auto ahead = [&]() {
    nq = nqd = nqdd = 0.0f;
    if (wk_jt(nw)) {
      const int j = wk_j(nw);
      nq = st.pos(j);
      if (dyn) {
        nqd = st.vel(j);
        nqdd = st.acc(j);
      }
    }
  };
  ahead();
  for (int i = 0; i <= total; ++i) {
    const bool end = i == total;
    const int pos = npos;
    const uint32_t w = nw;
    const int dep = end ? 0 : wk_dep(w);
    const float cq = nq, cqd = nqd, cqdd = nqdd;
    if (i + 1 < total) {
      npos = i + 1 < nrep ? wk.ancestor(sg.p0, sg.G, sg.g, i + 1) : sg.p0 + i + 1 - nrep;
      nw = wk(npos);
      ahead();
    }
    if (dyn) {
      while (sp > dep) close(--sp);
      flush();
    }
    if (end) break;
    sp = dep + 1;
    push(pos, w, i >= nrep, cq, cqd, cqdd);
  }
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
    float L[12], t[3];
    const int k = __ldg(r.chain + c), j = __ldg(r.jidx + k);
    local_xf(r, k, j >= 0 ? joint_var(r, k, st.pos(j)) : 0.0f, L, L + 9);
    if (c == c0) {
#pragma unroll
      for (int i = 0; i < 12; ++i) P[i] = L[i];
    } else {
      compose(P, L, t);
    }
  }
}

// parent pose from a link's world pose and its local transform: W <- W L^-1;
// t: the offset of the old origin from the new one
__device__ __forceinline__ void uncompose(float* W, const float* L, float* t) {
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    const float a = W[3 * i], b = W[3 * i + 1], c = W[3 * i + 2];
#pragma unroll
    for (int j = 0; j < 3; ++j)
      W[3 * i + j] = fmaf(c, L[3 * j + 2], fmaf(b, L[3 * j + 1], a * L[3 * j]));
  }
  rot(W, L + 9, t);
#pragma unroll
  for (int i = 0; i < 3; ++i) W[9 + i] -= t[i];
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
// added to o[15] = n, f, gw, gal, gA.  Four products with Io: it is rotated to the
// world once (45 operations, against 54 to rotate their arguments in and
// results out).
__device__ __forceinline__ void link_adjoint(const float* R, const float* I, const float* w,
                                             const float* al, const float* A, const float* wb,
                                             const float* ub, float* o) {
  float T[9], J[10], h[3];
#pragma unroll
  for (int i = 0; i < 3; ++i) rot_inertia(I, R + 3 * i, T + 3 * i);  // rows of R Io
  J[4] = dot3(T, R);
  J[5] = dot3(T + 3, R + 3);
  J[6] = dot3(T + 6, R + 6);
  J[7] = dot3(T, R + 3);
  J[8] = dot3(T, R + 6);
  J[9] = dot3(T + 3, R + 6);
  rot(R, I + 1, h);
  const float m = I[0];
  float Iw[3], c[3];
  rot_inertia(J, w, Iw);
  rot_inertia_acc(J, al, o);
  cross3_acc(w, Iw, o);
  cross3_acc(h, A, o);  // n
#pragma unroll
  for (int i = 0; i < 3; ++i) o[3 + i] = fmaf(m, A[i], o[3 + i]);
  cross3_acc(al, h, o + 3);
  centripetal_acc<1>(w, h, o + 3);  // f
  cross3(wb, w, c);
  rot_inertia_acc(J, c, o + 6);
  cross3_acc(Iw, wb, o + 6);
  centripetal_grad(w, h, ub, o + 6);  // gw
  rot_inertia_acc(J, wb, o + 9);
  cross3_acc(h, ub, o + 9);  // gal
#pragma unroll
  for (int i = 0; i < 3; ++i) o[12 + i] = fmaf(m, ub[i], o[12 + i]);
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
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(a), "l"(src) : "memory");
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
// OPT: what the sweep is compiled for (BwdOpt), so that a call that needs none
// of the rare options carries neither their branches nor their registers
// (humanoid48, every upstream gradient, 448-thread blocks: 0.097 -> 0.092 ms at 32768
// configurations, one thread a configuration 0.270 -> 0.260 ms at 99999).
enum BwdOpt {
  kBwdCost = 1,    // the fused cost (fc)
  kBwdRare = 2,    // external wrenches, joints that drive several links
  kBwdAny = 4,     // pose and sphere gradients as the arguments have them
  kBwdPose = 8,    // pose gradients, through the slots
  kBwdSphere = 16, // sphere gradients in runs of 4, through the slots
};
constexpr int kBwdGeneral = kBwdRare | kBwdAny;
constexpr int kBwdRows = kBwdPose | kBwdSphere;
// whether the sphere gradients g_sph of a robot can be read as float4 triples:
// its spheres come in runs of 4 (then b S + s is a multiple of 4) and the
// array is 16-byte aligned
__host__ __device__ __forceinline__ bool sphere_runs(const DevRobot& r, const float* g_sph) {
  return g_sph != nullptr && r.sph_vec4 && (reinterpret_cast<uintptr_t>(g_sph) & 15u) == 0;
}
// the fast instance that a call's arguments allow, else kBwdGeneral (wide:
// whether there is one for pose and sphere gradients together, or one for
// spheres alone)
inline int bwd_opt(const DevRobot& r, const BwdArgs& A, bool wide) {
  if (A.fext || A.g_fext || r.mimic_shared) return kBwdGeneral;
  if (A.g_sph && !sphere_runs(r, A.g_sph)) return kBwdGeneral;
  if (wide) return A.g_pose && A.g_sph ? kBwdRows : kBwdGeneral;
  return A.g_pose ? kBwdGeneral : A.g_sph ? kBwdSphere : 0;
}

// act: as for tree_fwd_seg.
template <int OPT, class WK, class St>
__device__ __forceinline__ float tree_bwd_seg(const DevRobot& r, const float4* rec, const WK& wk,
                                              const BwdArgs& A, const FusedCost& fc,
                                              const St& st, int64_t b, bool act, const Seg& sg,
                                              GradSlot gs = GradSlot{}) {
  constexpr bool FC = (OPT & kBwdCost) != 0, RARE = (OPT & kBwdRare) != 0;
  constexpr bool ANY = (OPT & kBwdAny) != 0;
  const int64_t B = A.B;
  float cost_part = 0.0f;
  const int n = r.n;
  BEnt stk[TMAXD];
  if (RARE && r.mimic_shared && act)
    for (int j = 0; j < r.d; ++j) {
      A.gq[(int64_t)j * B + b] = 0.0f;
      A.gqd[(int64_t)j * B + b] = 0.0f;
      A.gqdd[(int64_t)j * B + b] = 0.0f;
    }
  // the worst pair's gradient: u = g_dmin (c_i - c_j) / |c_i - c_j|, needed
  // only by the segment that owns one of the pair's links
  auto owned = [&](int k) {
    if (!sg.part) return true;
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
#pragma unroll
  for (int i = 0; i < 12; ++i) cW[i] = 0.0f;
#pragma unroll
  for (int i = 0; i < 3; ++i) cw[i] = cal[i] = cA[i] = cwb[i] = cub[i] = 0.0f;
#pragma unroll
  for (int i = 0; i < kSums; ++i) ps[i] = 0.0f;
  int pdep = -1;
  // bit e: entry e is an ancestor replayed for this segment (no own terms),
  // its acc holds children's sums
  uint32_t replayed = 0u, accv = 0u;
  int ckp = 0;  // the position the next close takes: the last pushed one, then parents
  auto sphere = [&](int s) { return WK::kSpheres ? rec[8 * n + s] : __ldg(r.sph + s); };
  const bool has_pose = ANY ? A.g_pose != nullptr : (OPT & kBwdPose) != 0;
  const bool sph4 = ANY ? sphere_runs(r, A.g_sph) : (OPT & kBwdSphere) != 0;
  const bool has_sph = ANY ? A.g_sph != nullptr : (OPT & kBwdSphere) != 0;
  const bool kin_grad = has_pose || has_sph;
  const bool use_slot = ANY ? gs.p != nullptr && kin_grad : kin_grad;
  auto issue = [&](const float4* q) {  // q: the link's record
    const float4 m = q[7];
    const int kn = __float_as_int(m.x);
    if (has_pose) {
      const float4* g4 = reinterpret_cast<const float4*>(A.g_pose + (b * n + (kn & 0xFF)) * 12);
      cp16(gs.p, g4);
      cp16(gs.p + gs.stride, g4 + 1);
      cp16(gs.p + 2 * gs.stride, g4 + 2);
    }
    if (sph4 && kn >= 256) {
      const float4* g4 =
          reinterpret_cast<const float4*>(A.g_sph + (b * r.S + __float_as_int(m.z)) * 3);
      cp16(gs.p + 3 * gs.stride, g4);
      cp16(gs.p + 4 * gs.stride, g4 + 1);
      cp16(gs.p + 5 * gs.stride, g4 + 2);
    }
    asm volatile("cp.async.commit_group;");
  };

  // gradient wrench of link k's kinematic outputs (pose, spheres, the worst
  // pair's spheres) in world axes about its origin: the points' gradients
  // join the rotation gradient G, whose wrench is the sum of the crosses of
  // R's columns with G's
  auto wrench = [&](const float4* q, float* w) {  // added to w
    const float4 m = q[7];
    const int kn = __float_as_int(m.x), k = kn & 0xFF, ns = kn >> 8, e0 = __float_as_int(m.w);
    float G[9];
#pragma unroll
    for (int i = 0; i < 9; ++i) G[i] = 0.0f;
    float* f = w + 3;
    // every owned link's rows were sent to the slot, at its push (a link closed
    // next) or at its last child's close
    const bool slot = use_slot;
    if (slot) asm volatile("cp.async.wait_group 0;" ::: "memory");
    if (has_pose) {
      const float4* g4 = reinterpret_cast<const float4*>(A.g_pose + (b * n + k) * 12);
      const float4 x0 = slot ? gs.p[0] : __ldg(g4), x1 = slot ? gs.p[gs.stride] : __ldg(g4 + 1),
                   x2 = slot ? gs.p[2 * gs.stride] : __ldg(g4 + 2);
      G[0] = x0.x; G[1] = x0.y; G[2] = x0.z; G[3] = x0.w; G[4] = x1.x;
      G[5] = x1.y; G[6] = x1.z; G[7] = x1.w; G[8] = x2.x;
      f[0] += x2.y; f[1] += x2.z; f[2] += x2.w;
    }
    if (sph4) {  // runs of 4 spheres: three float4 loads a run
      int s = __float_as_int(m.z);
      for (int e = 0; e < ns; e += 4) {
        if (e > 0) s = __ldg(r.ls_sph + e0 + e);
        const float4* g4 = reinterpret_cast<const float4*>(A.g_sph + (b * r.S + s) * 3);
        const bool fs = slot && e == 0;
        const float4 x0 = fs ? gs.p[3 * gs.stride] : __ldg(g4),
                     x1 = fs ? gs.p[4 * gs.stride] : __ldg(g4 + 1),
                     x2 = fs ? gs.p[5 * gs.stride] : __ldg(g4 + 2);
        const float gg[12] = {x0.x, x0.y, x0.z, x0.w, x1.x, x1.y, x1.z, x1.w, x2.x, x2.y, x2.z, x2.w};
#pragma unroll
        for (int i = 0; i < 4; ++i) point_grad(sphere(s + i), gg + 3 * i, G, f);
      }
    } else if (has_sph) {
      for (int e = 0; e < ns; ++e) {
        const int s = __ldg(r.ls_sph + e0 + e);
        const float* g = A.g_sph + (b * r.S + s) * 3;
        const float gg[3] = {__ldg(g), __ldg(g + 1), __ldg(g + 2)};
        point_grad(sphere(s), gg, G, f);
      }
    }
    if (k == pl1) point_grad(sphere(ps1), u, G, f);
    if (k == pl2) {
      const float mu[3] = {-u[0], -u[1], -u[2]};
      point_grad(sphere(ps2), mu, G, f);
    }
    const float* R = cW;
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      const float rc[3] = {R[j], R[3 + j], R[6 + j]}, gc[3] = {G[j], G[3 + j], G[6 + j]};
      cross3_acc(rc, gc, w);
    }
  };

  // post-order of the link at depth e; the registers hold its state; tgt:
  // the closes go on down to depth tgt
  auto close = [&](int e, int tgt) {
    const uint32_t w = wk(ckp);
    const float4* q = rec + 8 * ckp;
    ckp = wk_par(w);
    const int j = wk_j(w), jt = wk_jt(w);
    // the joint's state first: its loads' latency overlaps the own terms
    const float qj = jt ? st.pos(j) : 0.0f, vj = jt ? st.vel(j) : 0.0f, aj = jt ? st.acc(j) : 0.0f;
    const float tb = fresh ? ctb : stk[e].tb;
    const bool own = !((replayed >> e) & 1u);
    // the children's sums
    if (pdep != e) {
      if ((accv >> e) & 1u) {
#pragma unroll
        for (int i = 0; i < kSums; ++i) ps[i] = stk[e].acc[i];
      } else {
#pragma unroll
        for (int i = 0; i < kSums; ++i) ps[i] = 0.0f;
      }
    }
    pdep = -1;
    // plus the own terms (link_adjoint, minus the external wrench) and the
    // gradient wrench of the kinematic outputs
    if (own) {
      float I[10];
      rec_inertia(q, I);
      link_adjoint(cW, I, cw, cal, cA, cwb, cub, ps);
      const int k = __float_as_int(q[7].x) & 0xFF;
      if (RARE && A.fext) {
        const float* fe = A.fext + (b * n + k) * 6;
        const float xn[3] = {__ldg(fe), __ldg(fe + 1), __ldg(fe + 2)};
        const float xf[3] = {__ldg(fe + 3), __ldg(fe + 4), __ldg(fe + 5)};
        float t[3];
        rot(cW, xn, t);
#pragma unroll
        for (int i = 0; i < 3; ++i) ps[i] -= t[i];
        rot(cW, xf, t);
#pragma unroll
        for (int i = 0; i < 3; ++i) ps[3 + i] -= t[i];
      }
      if (kin_grad || k == pl1 || k == pl2) {
        wrench(q, ps + 15);
        // the next close's rows, while this one computes
        if (use_slot && e - 1 >= tgt && !((replayed >> (e - 1)) & 1u)) issue(rec + 8 * ckp);
      }
    }
    float *sn = ps, *sf = ps + 3, *gw = ps + 6, *gal = ps + 9, *gA = ps + 12, *Wn = ps + 15,
          *Wf = ps + 18;
    const float4 a4 = q[3];
    const float ax[3] = {a4.x, a4.y, a4.z};
    const float mm = a4.w;
    const float vq = mm * vj, aq = mm * aj;
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
    if (FC && jt) {
      float dqd = 0.0f, dqdd = 0.0f;  // the cost's direct gradients, once per joint
      if (own) {
        const int64_t at = (int64_t)j * B + b;
        const float tj = __ldg(fc.tau + at);
        dqd = 2.0f * (fc.length * vj + fc.e * (vj * tj) * tj);
        dqdd = 2.0f * fc.smooth * aj;
      }
      float* p0 = seg_part(sg, q, 0);
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
    } else if (jt) {
      float* p0 = seg_part(sg, q, 0);
      if (p0) {
        const size_t o = (size_t)sg.ns * sg.G * 32;
        p0[0] = mm * gq;
        p0[o] = mm * gqd;
        p0[2 * o] = mm * gqdd;
      } else {
        float* o0 = A.gq + (int64_t)j * B + b;
        float* o1 = A.gqd + (int64_t)j * B + b;
        float* o2 = A.gqdd + (int64_t)j * B + b;
        if (!RARE || !r.mimic_shared) {
          *o0 = mm * gq;
          *o1 = mm * gqd;
          *o2 = mm * gqdd;
        } else if (act) {
          *o0 += mm * gq;
          *o1 += mm * gqd;
          *o2 += mm * gqdd;
        }
      }
    }
    fresh = false;
    if (e > 0) {
      float L[12], rv[3];
      link_local<true>(q, w, qj, L);
      uncompose(cW, L, rv);
      cross3_sub(cal, rv, cA);
      centripetal_acc<-1>(cw, rv, cA);
      cross3_sub(cwb, rv, cub);
      // the sums about the parent's origin
      centripetal_grad(cw, rv, gA, gw);
      cross3_acc(rv, gA, gal);
      cross3_acc(rv, sf, sn);
      cross3_acc(rv, Wf, Wn);
      if ((accv >> (e - 1)) & 1u) {  // and the parent's from earlier children
        const BEnt& P = stk[e - 1];
        accv &= ~(1u << (e - 1));  // taken over by the pending registers
#pragma unroll
        for (int i = 0; i < kSums; ++i) ps[i] += P.acc[i];
      }
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

  // pre-order of the link at pos (the registers hold its parent's state);
  // own = false replays an ancestor of the segment (its own contributions are
  // zero); pq, pqd, pqdd, pgt: its joint's state and torque adjoint (FC: its
  // torque)
  auto push = [&](int pos, uint32_t w, bool own, float pq, float pqd, float pqdd, float pgt) {
    const float4* q = rec + 8 * pos;
    const int dep = wk_dep(w), jt = wk_jt(w), j = wk_j(w);
    float L[12];
    link_local<true>(q, w, pq, L);
    const float4 a4 = q[3];
    const float ax[3] = {a4.x, a4.y, a4.z};
    const float mm = a4.w;
    const float vq = mm * pqd, aq = mm * pqdd;
    // the adjoint of the force sweep's torque term: taubar of the joint
    float tb = 0.0f;
    if (FC) {
      if (jt) {  // the cost's torque gradient, as the cost kernel forms it
        const float t = pgt, l = __ldg(fc.lo + j), h = __ldg(fc.hi + j);
        const float v = pqd, a = pqdd;
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
      }
    } else {
      tb = mm * pgt;
    }
    // the link's state: pose, motion, and the torques' virtual motion
    // wb = wb_pa + s tb, ub = ub_pa + wb_pa x r (prismatic: ub + s tb)
    float s[3], rv[3], wp[3], alp[3], Ap[3];
    if (dep > 0) {
      compose(cW, L, rv);
      cross3_acc(cwb, rv, cub);
    } else {
#pragma unroll
      for (int i = 0; i < 12; ++i) cW[i] = L[i];
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        cw[i] = cal[i] = cwb[i] = cub[i] = rv[i] = 0.0f;
        cA[i] = r.abase[i];
      }
    }
    rot(cW, ax, s);
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      wp[i] = cw[i];
      alp[i] = cal[i];
      Ap[i] = cA[i];
    }
    joint_motion(jt, s, rv, vq, aq, wp, alp, Ap, cw, cal, cA);
    if (jt == 2) {
#pragma unroll
      for (int i = 0; i < 3; ++i) cub[i] = fmaf(s[i], tb, cub[i]);
    } else {
#pragma unroll
      for (int i = 0; i < 3; ++i) cwb[i] = fmaf(s[i], tb, cwb[i]);
    }
    ctb = tb;
    fresh = true;
    ckp = pos;
    const uint32_t bit = 1u << dep;
    accv &= ~bit;
    replayed = own ? (replayed & ~bit) : (replayed | bit);
    if (!wk_leaf(w)) stk[dep].tb = tb;
    if (RARE && own && A.g_fext) {  // dL/df_ext,k = -(wb, ub) in link coordinates
      float* o = A.g_fext + (b * n + (__float_as_int(q[7].x) & 0xFF)) * 6;
      float t[6];
      rotT(cW, cwb, t);
      rotT(cW, cub, t + 3);
#pragma unroll
      for (int i = 0; i < 6; ++i) o[i] = -t[i];
    }
  };

  // one loop over the replayed ancestors and the segment's links, as in the
  // forward
  const int nrep = wk_dep(wk(sg.p0)), total = nrep + sg.p1 - sg.p0;
  int sp = 0;
  int npos = wk.ancestor(sg.p0, sg.G, sg.g, 0);
  uint32_t nw = wk(npos);
  const float* const gt = FC ? fc.tau : A.g_tau;
  float nq = 0.0f, nqd = 0.0f, nqdd = 0.0f, ngt = 0.0f;
  auto fetch = [&](uint32_t w) {
    nq = nqd = nqdd = ngt = 0.0f;
    if (wk_jt(w)) {
      const int j = wk_j(w);
      nq = st.pos(j);
      nqd = st.vel(j);
      nqdd = st.acc(j);
      if (gt) ngt = __ldg(gt + (int64_t)j * B + b);
    }
  };
  for (int i = 0; i <= total; ++i) {
    const bool end = i == total, own = i >= nrep;
    const int pos = npos;
    const uint32_t w = nw;
    const int dep = end ? 0 : wk_dep(w);
    // this link's joint inputs, before the closes ahead of its push; the next
    // one's into L2 (held in registers a link ahead instead, the humanoid's
    // backward went 0.1025 -> 0.105 ms at 32768 configurations, 0.292 ->
    // 0.314 ms at 99999)
    if (!end) fetch(w);
    if (i + 1 < total) {
      npos = i + 1 < nrep ? wk.ancestor(sg.p0, sg.G, sg.g, i + 1) : sg.p0 + i + 1 - nrep;
      nw = wk(npos);
      if (wk_jt(nw)) {
        st.prefetch(wk_j(nw), true);
        if (gt) pf(gt + (int64_t)wk_j(nw) * B + b);
      }
    }
    while (sp > dep) close(--sp, dep);
    flush();
    if (end) break;
    sp = dep + 1;
    // a link closed right after its push (a leaf, or the segment's last
    // link): its rows start on their way now
    if (use_slot && own && (i + 1 >= total || wk_dep(nw) <= dep)) issue(rec + 8 * pos);
    push(pos, w, own, nq, nqd, nqdd, ngt);
  }
  if (use_slot) asm volatile("cp.async.wait_group 0;" ::: "memory");
  return cost_part;
}

}  // namespace wbe
