// k_tree.cu -- the single-robot depth-first sweep kernels (tree_sweep.cuh):
// one thread per configuration of a batch of B, or G warps per 32
// configurations (segmented sweep).
#include "tree_sweep.cuh"

#include <algorithm>

namespace wbe {

// Every sweep kernel stages the robot's link records (kRecWords floats a
// link: fixed transform, axis, mimic factors, inertia, output indices) once
// per block at the start of its shared memory: one base and constant offsets
// for everything a push or close reads of a link, in eight 16-byte loads, and
// out of the way of the depth-first stacks in L1.
constexpr size_t kSegSmemMax = 227 * 1024;  // dynamic shared memory of one block

// floats at the start of a backward block's shared memory: records, spheres
__host__ __device__ __forceinline__ size_t bwd_words(const DevRobot& r) {
  return kRecWords * (size_t)r.n + 4 * (size_t)r.S;
}

// levels of the forward's force stack (one less would hold: the deepest level never
// stores; but the fifth 128-thread block that then fits an SM takes its room from
// L1: humanoid, 99999 configurations in one segment, 0.190 -> 0.206 ms)
__host__ __device__ __forceinline__ size_t fs_levels(const DevRobot& r) {
  return (size_t)r.maxdepth;
}

// this thread's warp, known to be the same for its whole warp
__device__ __forceinline__ int warp_of() { return __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0); }

// the block's dynamic shared memory covers `words` floats
__device__ __forceinline__ bool smem_holds(size_t words) {
  unsigned dyn;
  asm("mov.u32 %0, %%dynamic_smem_size;" : "=r"(dyn));
  return sizeof(float) * words <= dyn;
}

// the configuration b of this lane in the warp whose first is b0 (act); a lane
// past the end takes the last one and act = false; false: the warp has none
__device__ __forceinline__ bool own_config(int64_t B, int64_t b0, int64_t* b, bool* act) {
  if (b0 >= B) return false;
  const int64_t own = b0 + (threadIdx.x & 31);
  *act = own < B;
  *b = *act ? own : B - 1;
  return true;
}

// MODE kFwdShared: the force stack in shared memory behind the link records,
// as in the segmented forward below
template <int MODE>
__device__ __forceinline__ void fwd_block(const DevRobot& r, const WalkTab& wt, const FwdArgs& A,
                                          float4* rec) {
  constexpr bool FS = MODE == kFwdShared;
  float* sm = reinterpret_cast<float*>(rec) + kRecWords * (size_t)r.n;
  if (FS && !smem_holds(kRecWords * (size_t)r.n + 6 * fs_levels(r) * blockDim.x)) return;
  stage_recs(r, -1, rec, threadIdx.x, blockDim.x);
  __syncthreads();
  int64_t b;
  bool act;
  if (!own_config(A.B, blockIdx.x * (int64_t)blockDim.x + 32 * warp_of(), &b, &act)) return;
  Seg sg = whole_sweep(r);
  if (FS) {
    sg.fst = reinterpret_cast<float2*>(sm) + threadIdx.x;
    sg.fstr = blockDim.x;
  }
  tree_fwd_seg<MODE>(r, rec, ConstWalk<true>{wt}, A, ArrayStates{A.q, A.qd, A.qdd, A.B, b}, b, act, sg);
}
template <int MODE>
__global__ void __launch_bounds__(256) tree_fwd_kernel(const __grid_constant__ DevRobot r,
                                                       const __grid_constant__ WalkTab wt,
                                                       const __grid_constant__ FwdArgs A) {
  extern __shared__ float4 rec[];
  fwd_block<MODE>(r, wt, A, rec);
}
// The same for robots without branches, capped at 72 registers: 28 warps an SM
// where 78 allow 24, at the price of spills (fwd_chain: when it is taken).  The
// sweep is latency-bound and a chain never touches the branch stack.  7-DoF arm,
// 131072 configurations: 0.0280 -> 0.0249 ms (64 registers: 0.0293; the branch code
// compiled out besides: 0.0263).
__global__ void __maxnreg__(72) tree_fwd_chain_kernel(const __grid_constant__ DevRobot r,
                                                      const __grid_constant__ WalkTab wt,
                                                      const __grid_constant__ FwdArgs A) {
  extern __shared__ float4 rec[];
  fwd_block<kFwdShared>(r, wt, A, rec);
}

// The backward sweeps are capped at 128 registers (two 256-thread blocks per
// SM, or one 512-thread block of a segmented sweep): more a thread cost the
// occupancy that hides each link's chain, fewer (104) spilled and were 2 %
// slower at the same number of resident warps.  The segmented sweeps take blocks of up to
// 512 threads, so that one block per SM holds the staged link parameters once
// and the shared-memory carveout stays small.
template <int OPT>
__global__ void __launch_bounds__(256, 2) tree_bwd_kernel(const __grid_constant__ DevRobot r,
                                                          const __grid_constant__ WalkTab wt,
                                                          const __grid_constant__ BwdArgs A) {
  extern __shared__ float4 rec[];
  stage_recs(r, -1, rec, threadIdx.x, blockDim.x);
  stage_spheres(r, rec);
  __syncthreads();
  int64_t b;
  bool act;
  if (!own_config(A.B, blockIdx.x * (int64_t)blockDim.x + 32 * warp_of(), &b, &act)) return;
  const GradSlot gs = grad_slot_of(reinterpret_cast<float*>(rec) + bwd_words(r));
  tree_bwd_seg<OPT>(r, rec, ConstWalk<false>{wt}, A, FusedCost{},
                      ArrayStates{A.q, A.qd, A.qdd, A.B, b}, b, act, whole_sweep(r), gs);
}

// Segmented sweeps, plan t (G = 2 << t segments).  A block holds CG groups of
// G warps; warp w sweeps segment w % G of the 32 configurations of group
// w / G.  Shared memory per group: the partial outputs [nout][ns][G][32] of
// the ns links that several segments hold, summed in segment order after the
// barrier by the group's warps (slot s by warp s % G).
__device__ __forceinline__ Seg seg_of(const DevRobot& r, int t, int g, float* part) {
  return Seg{r.seg_pos[t][g], r.seg_pos[t][g + 1], g, 2 << t, part, r.seg_ns[t],
             (int)(threadIdx.x & 31)};
}

// MODE kFwdShared: the force stack in shared memory, [fs_levels][3][threads] float2 behind
// the partials (a link's F is stored when its first child is pushed
// and read back at that child's close; in local memory these round trips
// missed L1 61 % of the time)
template <int MODE>
__global__ void __launch_bounds__(512) tree_fwd_seg_kernel(const __grid_constant__ DevRobot r,
                                                           const __grid_constant__ WalkTab wt,
                                                           const __grid_constant__ FwdArgs A,
                                                           int t) {
  extern __shared__ float4 rec[];
  float* part = reinterpret_cast<float*>(rec) + kRecWords * (size_t)r.n;
  const int G = 2 << t;
  const int CG = blockDim.x / (32 * G);
  const int wid = warp_of(), cg = wid / G;
  const int ns = r.seg_ns[t];
  // the launch reserves the stack for this block's threads; a block that
  // finds less shared memory than that does nothing (its outputs stay
  // unwritten) instead of indexing past it
  if (MODE == kFwdShared && !smem_holds((size_t)CG * ns * G * 32 + kRecWords * (size_t)r.n +
                        6 * fs_levels(r) * blockDim.x))
    return;
  Seg sg = seg_of(r, t, wid % G, part + (size_t)cg * ns * G * 32);
  for (int s = 0; s < ns; ++s) sg.part[(s * G + sg.g) * 32 + sg.lane] = 0.0f;
  stage_recs(r, t, rec, threadIdx.x, blockDim.x);
  if (MODE == kFwdShared) {
    sg.fst = reinterpret_cast<float2*>(part + (size_t)CG * ns * G * 32) + threadIdx.x;
    sg.fstr = blockDim.x;
  }
  __syncthreads();
  int64_t b;
  bool act = false;
  if (own_config(A.B, ((int64_t)blockIdx.x * CG + cg) * 32, &b, &act))
    tree_fwd_seg<MODE>(r, rec, ConstWalk<true>{wt}, A, ArrayStates{A.q, A.qd, A.qdd, A.B, b}, b, act, sg);
  __syncthreads();
  if (act && A.tau) {
    for (int s = sg.g; s < ns; s += G) {
      float acc = 0.0f;
      for (int h = 0; h < G; ++h) acc += sg.part[(s * G + h) * 32 + sg.lane];
      const int k = __ldg(r.seg_slot_link + t * r.n + s);
      A.tau[(int64_t)__ldg(r.jidx + k) * A.B + b] = acc;
    }
  }
}

template <int OPT>
__global__ void __launch_bounds__(512, 1) tree_bwd_seg_kernel(const __grid_constant__ DevRobot r,
                                                           const __grid_constant__ WalkTab wt,
                                                           const __grid_constant__ BwdArgs A,
                                                           int t) {
  extern __shared__ float4 rec[];
  float* part = reinterpret_cast<float*>(rec) + bwd_words(r);
  const int G = 2 << t;
  const int CG = blockDim.x / (32 * G);
  const int wid = warp_of(), cg = wid / G;
  const int ns = r.seg_ns[t];
  const size_t o = (size_t)ns * G * 32;  // one output's partials
  Seg sg = seg_of(r, t, wid % G, part + (size_t)cg * 3 * o);
  for (int s = 0; s < ns; ++s)
    for (int q = 0; q < 3; ++q) sg.part[q * o + (s * G + sg.g) * 32 + sg.lane] = 0.0f;
  stage_recs(r, t, rec, threadIdx.x, blockDim.x);
  stage_spheres(r, rec);
  // the gradient-row slots behind the partials (reserved by the launch when
  // there are upstream pose or sphere gradients)
  const GradSlot gs = grad_slot_of(part + (size_t)CG * 3 * o);
  __syncthreads();
  int64_t b;
  bool act = false;
  if (own_config(A.B, ((int64_t)blockIdx.x * CG + cg) * 32, &b, &act))
    tree_bwd_seg<OPT>(r, rec, ConstWalk<false>{wt}, A, FusedCost{},
                        ArrayStates{A.q, A.qd, A.qdd, A.B, b}, b, act, sg, gs);
  __syncthreads();
  if (act) {
    for (int s = sg.g; s < ns; s += G) {
      float acc[3] = {0.0f, 0.0f, 0.0f};
      for (int h = 0; h < G; ++h)
        for (int q = 0; q < 3; ++q) acc[q] += sg.part[q * o + (s * G + h) * 32 + sg.lane];
      const int k = __ldg(r.seg_slot_link + t * r.n + s);
      const int64_t at = (int64_t)__ldg(r.jidx + k) * A.B + b;
      A.gq[at] = acc[0];
      A.gqd[at] = acc[1];
      A.gqdd[at] = acc[2];
    }
  }
}

// a configuration's cost: its joints' terms, then the collision term
__device__ __forceinline__ float total_cost(const FusedCost& fc, int64_t b, float c) {
  return fc.d_min ? fmaf(fc.w, fmaxf(0.0f, -__ldg(fc.d_min + b)), c) : c;
}

// The same sweeps with the trajectory cost in their prologue (FusedCost):
// separate kernels, so that the plain ones keep their register allocation.
// The segmented one adds each configuration's cost terms over the segments
// in segment order (deterministic) after the barrier.
template <int OPT>
__global__ void __launch_bounds__(256, 2) tree_bwd_cost_kernel(
    const __grid_constant__ DevRobot r, const __grid_constant__ WalkTab wt,
    const __grid_constant__ BwdArgs A, const __grid_constant__ FusedCost fc) {
  extern __shared__ float4 rec[];
  stage_recs(r, -1, rec, threadIdx.x, blockDim.x);
  stage_spheres(r, rec);
  __syncthreads();
  int64_t b;
  bool act;
  if (!own_config(A.B, blockIdx.x * (int64_t)blockDim.x + 32 * warp_of(), &b, &act)) return;
  const GradSlot gs = grad_slot_of(reinterpret_cast<float*>(rec) + bwd_words(r));
  const float c = tree_bwd_seg<kBwdCost | OPT>(r, rec, ConstWalk<false>{wt}, A, fc,
                                     ArrayStates{A.q, A.qd, A.qdd, A.B, b}, b, act,
                                     whole_sweep(r), gs);
  if (fc.cost) fc.cost[b] = total_cost(fc, b, c);
}

template <int OPT>
__global__ void __launch_bounds__(512, 1) tree_bwd_cost_seg_kernel(
    const __grid_constant__ DevRobot r, const __grid_constant__ WalkTab wt,
    const __grid_constant__ BwdArgs A, const __grid_constant__ FusedCost fc, int t) {
  extern __shared__ float4 rec[];
  float* part = reinterpret_cast<float*>(rec) + bwd_words(r);
  const int G = 2 << t;
  const int CG = blockDim.x / (32 * G);
  const int wid = warp_of(), cg = wid / G;
  const int ns = r.seg_ns[t];
  const size_t o = (size_t)ns * G * 32;  // one output's partials
  Seg sg = seg_of(r, t, wid % G, part + (size_t)cg * (3 * o + G * 32));
  float* cpart = sg.part + 3 * o;  // [G][32] the segments' cost terms
  for (int s = 0; s < ns; ++s)
    for (int q = 0; q < 3; ++q) sg.part[q * o + (s * G + sg.g) * 32 + sg.lane] = 0.0f;
  stage_recs(r, t, rec, threadIdx.x, blockDim.x);
  stage_spheres(r, rec);
  const GradSlot gs = grad_slot_of(part + (size_t)CG * (3 * o + G * 32));
  __syncthreads();
  int64_t b;
  bool act = false;
  float c = 0.0f;
  if (own_config(A.B, ((int64_t)blockIdx.x * CG + cg) * 32, &b, &act))
    c = tree_bwd_seg<kBwdCost | OPT>(r, rec, ConstWalk<false>{wt}, A, fc,
                           ArrayStates{A.q, A.qd, A.qdd, A.B, b}, b, act, sg, gs);
  cpart[sg.g * 32 + sg.lane] = c;
  __syncthreads();
  if (act && sg.g == 0 && fc.cost) {
    float acc = 0.0f;
    for (int h = 0; h < G; ++h) acc += cpart[h * 32 + sg.lane];
    fc.cost[b] = total_cost(fc, b, acc);
  }
  if (act) {
    for (int s = sg.g; s < ns; s += G) {
      float acc[3] = {0.0f, 0.0f, 0.0f};
      for (int h = 0; h < G; ++h)
        for (int q = 0; q < 3; ++q) acc[q] += sg.part[q * o + (s * G + h) * 32 + sg.lane];
      const int k = __ldg(r.seg_slot_link + t * r.n + s);
      const int64_t at = (int64_t)__ldg(r.jidx + k) * A.B + b;
      A.gq[at] = acc[0];
      A.gqd[at] = acc[1];
      A.gqdd[at] = acc[2];
    }
  }
}

// The sweeps with the joint states evaluated from B-spline control points
// where they need them (SplineStates): no state arrays are read or written.
// Each thread keeps its sample's basis rows in shared memory, in front of the
// segments' partials.
__device__ __forceinline__ SplineStates spline_states(const DevRobot& r, const SplineArgs& sp,
                                                      int64_t b, float* bs) {
  const int64_t tr = b / sp.T;
  int k;
  float al;
  bs_sample((int)(b - tr * sp.T), sp.K, sp.T, k, al);
  float Bm[3][4];
  bs_basis(al, sp.dt, Bm);
#pragma unroll
  for (int q = 0; q < 3; ++q)
#pragma unroll
    for (int l = 0; l < 4; ++l) bs[4 * q + l] = Bm[q][l];
  return SplineStates{sp.U + (tr * r.d) * sp.K + k, sp.K, bs};
}

template <int MODE>
__global__ void __launch_bounds__(256) tree_fwd_spline_kernel(
    const __grid_constant__ DevRobot r, const __grid_constant__ WalkTab wt,
    const __grid_constant__ FwdArgs A, const __grid_constant__ SplineArgs sp) {
  extern __shared__ float4 rec[];
  float* sm = reinterpret_cast<float*>(rec) + kRecWords * (size_t)r.n;
  stage_recs(r, -1, rec, threadIdx.x, blockDim.x);
  __syncthreads();
  int64_t b;
  bool act;
  if (!own_config(A.B, blockIdx.x * (int64_t)blockDim.x + 32 * warp_of(), &b, &act)) return;
  const SplineStates st = spline_states(r, sp, b, sm + 12 * threadIdx.x);
  tree_fwd_seg<MODE>(r, rec, ConstWalk<true>{wt}, A, st, b, act, whole_sweep(r));
}

// MODE as for tree_fwd_seg_kernel; the force stack follows the partials
template <int MODE>
__global__ void __launch_bounds__(512) tree_fwd_spline_seg_kernel(
    const __grid_constant__ DevRobot r, const __grid_constant__ WalkTab wt,
    const __grid_constant__ FwdArgs A, const __grid_constant__ SplineArgs sp, int t) {
  extern __shared__ float4 rec[];
  float* sm = reinterpret_cast<float*>(rec) + kRecWords * (size_t)r.n;
  float* part = sm + 12 * blockDim.x;
  const int G = 2 << t;
  const int CG = blockDim.x / (32 * G);
  const int wid = warp_of(), cg = wid / G;
  const int ns = r.seg_ns[t];
  if (MODE == kFwdShared && !smem_holds(12 * (size_t)blockDim.x + (size_t)CG * ns * G * 32 +
                        kRecWords * (size_t)r.n + 6 * fs_levels(r) * blockDim.x))
    return;
  Seg sg = seg_of(r, t, wid % G, part + (size_t)cg * ns * G * 32);
  for (int s = 0; s < ns; ++s) sg.part[(s * G + sg.g) * 32 + sg.lane] = 0.0f;
  stage_recs(r, t, rec, threadIdx.x, blockDim.x);
  if (MODE == kFwdShared) {
    sg.fst = reinterpret_cast<float2*>(part + (size_t)CG * ns * G * 32) + threadIdx.x;
    sg.fstr = blockDim.x;
  }
  __syncthreads();
  int64_t b;
  bool act = false;
  if (own_config(A.B, ((int64_t)blockIdx.x * CG + cg) * 32, &b, &act))
    tree_fwd_seg<MODE>(r, rec, ConstWalk<true>{wt}, A, spline_states(r, sp, b, sm + 12 * threadIdx.x), b,
                     act, sg);
  __syncthreads();
  if (act && A.tau) {
    for (int s = sg.g; s < ns; s += G) {
      float acc = 0.0f;
      for (int h = 0; h < G; ++h) acc += sg.part[(s * G + h) * 32 + sg.lane];
      const int k = __ldg(r.seg_slot_link + t * r.n + s);
      A.tau[(int64_t)__ldg(r.jidx + k) * A.B + b] = acc;
    }
  }
}

template <int OPT>
__global__ void __launch_bounds__(256, 2) tree_bwd_spline_cost_kernel(
    const __grid_constant__ DevRobot r, const __grid_constant__ WalkTab wt,
    const __grid_constant__ BwdArgs A, const __grid_constant__ FusedCost fc,
    const __grid_constant__ SplineArgs sp) {
  extern __shared__ float4 rec[];
  float* sm = reinterpret_cast<float*>(rec) + bwd_words(r);
  stage_recs(r, -1, rec, threadIdx.x, blockDim.x);
  stage_spheres(r, rec);
  __syncthreads();
  int64_t b;
  bool act;
  if (!own_config(A.B, blockIdx.x * (int64_t)blockDim.x + 32 * warp_of(), &b, &act)) return;
  const GradSlot gs = grad_slot_of(sm + 12 * blockDim.x);
  const float c = tree_bwd_seg<kBwdCost | OPT>(r, rec, ConstWalk<false>{wt}, A, fc,
                                               spline_states(r, sp, b, sm + 12 * threadIdx.x), b,
                                               act, whole_sweep(r), gs);
  if (fc.cost) fc.cost[b] = total_cost(fc, b, c);
}

template <int OPT>
__global__ void __launch_bounds__(512, 1) tree_bwd_spline_cost_seg_kernel(
    const __grid_constant__ DevRobot r, const __grid_constant__ WalkTab wt,
    const __grid_constant__ BwdArgs A, const __grid_constant__ FusedCost fc,
    const __grid_constant__ SplineArgs sp, int t) {
  extern __shared__ float4 rec[];
  float* sm = reinterpret_cast<float*>(rec) + bwd_words(r);
  float* base = sm + 12 * blockDim.x;
  const int G = 2 << t;
  const int CG = blockDim.x / (32 * G);
  const int wid = warp_of(), cg = wid / G;
  const int ns = r.seg_ns[t];
  const size_t o = (size_t)ns * G * 32;  // one output's partials
  Seg sg = seg_of(r, t, wid % G, base + (size_t)cg * (3 * o + G * 32));
  float* cpart = sg.part + 3 * o;  // [G][32] the segments' cost terms
  for (int s = 0; s < ns; ++s)
    for (int q = 0; q < 3; ++q) sg.part[q * o + (s * G + sg.g) * 32 + sg.lane] = 0.0f;
  stage_recs(r, t, rec, threadIdx.x, blockDim.x);
  stage_spheres(r, rec);
  const GradSlot gs = grad_slot_of(base + (size_t)CG * (3 * o + G * 32));
  __syncthreads();
  int64_t b;
  bool act = false;
  float c = 0.0f;
  if (own_config(A.B, ((int64_t)blockIdx.x * CG + cg) * 32, &b, &act))
    c = tree_bwd_seg<kBwdCost | OPT>(r, rec, ConstWalk<false>{wt}, A, fc,
                           spline_states(r, sp, b, sm + 12 * threadIdx.x), b, act, sg, gs);
  cpart[sg.g * 32 + sg.lane] = c;
  __syncthreads();
  if (act && sg.g == 0 && fc.cost) {
    float acc = 0.0f;
    for (int h = 0; h < G; ++h) acc += cpart[h * 32 + sg.lane];
    fc.cost[b] = total_cost(fc, b, acc);
  }
  if (act) {
    for (int s = sg.g; s < ns; s += G) {
      float acc[3] = {0.0f, 0.0f, 0.0f};
      for (int h = 0; h < G; ++h)
        for (int q = 0; q < 3; ++q) acc[q] += sg.part[q * o + (s * G + h) * 32 + sg.lane];
      const int k = __ldg(r.seg_slot_link + t * r.n + s);
      const int64_t at = (int64_t)__ldg(r.jidx + k) * A.B + b;
      A.gq[at] = acc[0];
      A.gqd[at] = acc[1];
      A.gqdd[at] = acc[2];
    }
  }
}

static size_t rec_smem(const DevRobot& r, bool fwd) {
  return sizeof(float) * (fwd ? kRecWords * (size_t)r.n : bwd_words(r));
}

static int seg_plan(int segments) { return segments == 2 ? 0 : segments == 4 ? 1 : 2; }
static int seg_groups(int segments, int threads) { return std::max(1, threads / (32 * segments)); }

// per group of G warps: the shared-slot partials of each output (tau in the
// forward; gq, gqd, gqdd in the backward), plus, for the cost variant, one
// cost term per segment; per block, the staged link records
size_t tree_seg_smem(const DevRobot& r, int segments, int threads, bool fwd, bool cost) {
  const int t = seg_plan(segments);
  const size_t per =
      (size_t)(fwd ? 1 : 3) * r.seg_ns[t] * segments * 32 + (cost ? segments * 32 : 0);
  return (size_t)seg_groups(segments, threads) * per * sizeof(float) + rec_smem(r, fwd);
}

// a backward block's gradient-row slots (GradSlot), when it has upstream pose
// or sphere gradients to read
size_t grad_slot_smem(int segments, int threads) {
  return 16 + (size_t)kGradSlotBytes * 32 * segments * seg_groups(segments, threads);
}

template <class Args>
static cudaError_t launch_seg(void (*kern)(DevRobot, WalkTab, Args, int), const DevRobot& r,
                              const WalkTab& wt, const Args& a, int threads, int segments, bool fwd, size_t extra,
                              cudaStream_t s) {
  const int t = seg_plan(segments);
  const int CG = seg_groups(segments, threads);
  const size_t smem = tree_seg_smem(r, segments, threads, fwd, false) + extra;
  cudaError_t e =
      allow_smem((const void*)kern, smem);
  if (e != cudaSuccess) return e;
  fit_carveout((const void*)kern, 32 * segments * CG, smem);
  const int64_t groups = (a.B + 31) / 32;
  const int64_t grid = (groups + CG - 1) / CG;
  kern<<<(unsigned)grid, 32 * segments * CG, smem, s>>>(r, wt, a, t);
  return cudaGetLastError();
}

// A backward launch's kernel, its dynamic shared memory and its carveout; the
// arguments then follow in launch order.
template <class... P, class... V>
static cudaError_t launch_bwd(void (*kern)(P...), int64_t B, int groups, int block, size_t smem,
                              cudaStream_t s, const V&... v) {
  cudaError_t e =
      allow_smem((const void*)kern, smem);
  if (e != cudaSuccess) return e;
  fit_carveout((const void*)kern, block, smem);
  const int64_t grid = ((B + 31) / 32 + groups - 1) / groups;
  kern<<<(unsigned)grid, block, smem, s>>>(v...);
  return cudaGetLastError();
}

// Dynamic shared memory of a block of G segments that writes poses only.  Its 46 or 48
// registers a thread allow 40 warps an SM, whose lanes each write 48 bytes at a time
// into rows of their own (G places of a row at once); when the poses no longer fit
// the L2 (129 MB) it evicts lines that are not yet full.  So batches of more than 20
// warps an SM then have at most 16 at a time: humanoid, 131072 configurations (308
// MB) 0.239 -> 0.195 ms (12 warps the same, 20 0.201), 23-DoF (150 MB) 0.118 -> 0.093;
// 99999 configurations 0.171 -> 0.155 and, at 110 MB in two segments, 0.081 -> 0.064.
// Smaller poses are better off without (20 links, 110 MB: 0.041 ms), and so are up to
// 20 warps (32 links, 80000 configurations 0.068 and 0.073).
bool poses_beyond_l2(const DevRobot& r, int64_t B, int G) {
  return B * r.n * 48 > (int64_t)(G > 1 ? 100 : 112) << 20;
}
static size_t pose_smem(const DevRobot& r, int64_t B, int G, int threads, size_t smem) {
  const int64_t warps = (B + 31) / 32 * G;
  if (!poses_beyond_l2(r, B, G) || warps <= 20LL * sm_count()) return smem;
  const size_t blocks = std::max(1, 16 * 32 / threads);
  const size_t share = 228 * 1024 / blocks - 1024;  // 228 KB an SM, 1 KB of it each block's own
  return std::max(smem, std::min(kSegSmemMax, share));
}

// Whether the chain kernel is the better one: where the batch has more warps an SM
// than the general kernel's registers hold and the force stacks of its blocks leave
// the shared memory for more (21 KB a 128-thread block for 7 links do; 37 KB for 12
// do not, nor do the humanoid's 46).  Elsewhere the spills are all it brings: 12, 20
// and 32 links, 131072 configurations 0.058, 0.124, 0.291 ms against 0.040, 0.101,
// 0.193; the arm's 99999 configurations 0.0209 and 0.0182.
static cudaError_t fwd_chain(const DevRobot& r, int64_t B, int threads, size_t smem, bool* out) {
  *out = false;
  if (r.maxdepth != r.n) return cudaSuccess;  // a link a level: no branches
  const void* kerns[2] = {(const void*)tree_fwd_kernel<kFwdShared>,
                          (const void*)tree_fwd_chain_kernel};
  int blocks[2] = {0, 0};
  for (int i = 0; i < 2; ++i) {
    cudaError_t e = allow_smem(kerns[i], smem);
    if (e == cudaSuccess) e = max_blocks(kerns[i], threads, smem, &blocks[i]);
    if (e != cudaSuccess) return e;
  }
  *out = blocks[1] > blocks[0] && B > (int64_t)blocks[0] * threads * sm_count();
  return cudaSuccess;
}

// The one-segment forward sweep's kernel and dynamic shared memory.
struct WholeKernel {
  void (*kern)(DevRobot, WalkTab, FwdArgs);
  size_t smem;
};
static cudaError_t fwd_whole(const DevRobot& r, int64_t B, int threads, bool tau, WholeKernel* out) {
  const size_t fs = sizeof(float) * 6 * fs_levels(r) * threads;  // the force stack
  const bool use_fs = tau && rec_smem(r, true) + fs <= kSegSmemMax;
  size_t smem = rec_smem(r, true) + (use_fs ? fs : 0);
  if (!tau) smem = pose_smem(r, B, 1, threads, smem);
  bool chain = false;
  const cudaError_t e = use_fs ? fwd_chain(r, B, threads, smem, &chain) : cudaSuccess;
  out->kern = chain    ? tree_fwd_chain_kernel
              : use_fs ? tree_fwd_kernel<kFwdShared>
              : tau    ? tree_fwd_kernel<kFwdLocal>
                       : tree_fwd_kernel<kFwdPose>;
  out->smem = smem;
  return e;
}
static size_t fwd_spline_smem(const DevRobot& r, int64_t B, int threads, bool tau) {
  const size_t smem = 12 * sizeof(float) * threads + rec_smem(r, true);
  return tau ? smem : pose_smem(r, B, 1, threads, smem);
}

// the blocks of `threads` threads that an SM holds of it (spline: with states from
// control points)
cudaError_t fwd_whole_blocks(const DevRobot& r, int64_t B, int threads, bool tau, bool spline,
                             int* out) {
  const void* kern;
  size_t smem;
  if (spline) {
    kern = tau ? (const void*)tree_fwd_spline_kernel<kFwdLocal>
               : (const void*)tree_fwd_spline_kernel<kFwdPose>;
    smem = fwd_spline_smem(r, B, threads, tau);
  } else {
    WholeKernel w;
    const cudaError_t e = fwd_whole(r, B, threads, tau, &w);
    if (e != cudaSuccess) return e;
    kern = (const void*)w.kern;
    smem = w.smem;
  }
  const cudaError_t e = allow_smem(kern, smem);
  return e != cudaSuccess ? e : max_blocks(kern, threads, smem, out);
}

cudaError_t launch_tree_fwd(const DevRobot& r, const WalkTab& wt, const FwdArgs& a, int threads, int segments,
                            cudaStream_t s) {
  if (threads <= 0) threads = 128;
  if (segments > 1) {
    // the force stack in shared memory when it fits one block's limit (the
    // humanoid's 13 levels x 448 threads: 140 KB; forward 0.0835 ->
    // 0.0809 ms), else in local memory
    const size_t bt = (size_t)32 * segments * seg_groups(segments, threads);
    const size_t fs = sizeof(float) * 6 * fs_levels(r) * bt;
    if (a.tau && tree_seg_smem(r, segments, threads, true, false) + fs <= kSegSmemMax)
      return launch_seg(tree_fwd_seg_kernel<kFwdShared>, r, wt, a, threads, segments, true, fs, s);
    const size_t base = tree_seg_smem(r, segments, threads, true, false);
    return launch_seg(a.tau ? tree_fwd_seg_kernel<kFwdLocal> : tree_fwd_seg_kernel<kFwdPose>, r, wt,
                      a, threads, segments, true,
                      a.tau ? 0 : pose_smem(r, a.B, segments, (int)bt, base) - base, s);
  }
  WholeKernel w;
  cudaError_t e = fwd_whole(r, a.B, threads, a.tau != nullptr, &w);
  if (e == cudaSuccess) e = allow_smem((const void*)w.kern, w.smem);
  if (e != cudaSuccess) return e;
  fit_carveout((const void*)w.kern, threads, w.smem);
  const int64_t grid = (a.B + threads - 1) / threads;
  w.kern<<<(unsigned)grid, threads, w.smem, s>>>(r, wt, a);
  return cudaGetLastError();
}

cudaError_t launch_tree_bwd(const DevRobot& r, const WalkTab& wt, const BwdArgs& a, int threads,
                            int segments, cudaStream_t s, const FusedCost* fc) {
  if (threads <= 0) threads = 128;
  const int opt = bwd_opt(r, a, fc == nullptr);
  const int CG = segments > 1 ? seg_groups(segments, threads) : threads / 32;
  const int block = 32 * segments * CG;
  const size_t smem = (segments > 1 ? tree_seg_smem(r, segments, threads, false, fc != nullptr)
                                    : rec_smem(r, false)) +
                      (a.g_pose || a.g_sph ? grad_slot_smem(segments, threads) : 0);
  if (segments > 1) {
    const int t = seg_plan(segments);
    if (!fc)
      return launch_bwd(opt == kBwdRows ? tree_bwd_seg_kernel<kBwdRows>
                                        : tree_bwd_seg_kernel<kBwdGeneral>,
                        a.B, CG, block, smem, s, r, wt, a, t);
    return launch_bwd(opt == 0            ? tree_bwd_cost_seg_kernel<0>
                      : opt == kBwdSphere ? tree_bwd_cost_seg_kernel<kBwdSphere>
                                          : tree_bwd_cost_seg_kernel<kBwdGeneral>,
                      a.B, CG, block, smem, s, r, wt, a, *fc, t);
  }
  if (!fc)
    return launch_bwd(opt == kBwdRows ? tree_bwd_kernel<kBwdRows> : tree_bwd_kernel<kBwdGeneral>,
                      a.B, CG, block, smem, s, r, wt, a);
  return launch_bwd(opt == 0            ? tree_bwd_cost_kernel<0>
                    : opt == kBwdSphere ? tree_bwd_cost_kernel<kBwdSphere>
                                        : tree_bwd_cost_kernel<kBwdGeneral>,
                    a.B, CG, block, smem, s, r, wt, a, *fc);
}

cudaError_t launch_tree_fwd_spline(const DevRobot& r, const WalkTab& wt, const FwdArgs& a, const SplineArgs& sp,
                                   int threads, int segments, cudaStream_t s) {
  if (threads <= 0) threads = 128;
  if (segments > 1) {
    const int t = seg_plan(segments);
    const int CG = seg_groups(segments, threads);
    const int block = 32 * segments * CG;
    const size_t base = tree_seg_smem(r, segments, threads, true, false) + 12 * sizeof(float) * block;
    const size_t fs = sizeof(float) * 6 * fs_levels(r) * block;  // the force stack
    const bool use_fs = a.tau && base + fs <= kSegSmemMax;
    const size_t smem = use_fs ? base + fs : a.tau ? base : pose_smem(r, a.B, segments, block, base);
    auto kern = use_fs ? tree_fwd_spline_seg_kernel<kFwdShared>
                : a.tau ? tree_fwd_spline_seg_kernel<kFwdLocal>
                        : tree_fwd_spline_seg_kernel<kFwdPose>;
    cudaError_t e =
        allow_smem((const void*)kern, smem);
    if (e != cudaSuccess) return e;
    fit_carveout((const void*)kern, block, smem);
    const int64_t grid = ((a.B + 31) / 32 + CG - 1) / CG;
    kern<<<(unsigned)grid, block, smem, s>>>(r, wt, a, sp, t);
    return cudaGetLastError();
  }
  const size_t smem = fwd_spline_smem(r, a.B, threads, a.tau != nullptr);
  auto kern = a.tau ? tree_fwd_spline_kernel<kFwdLocal> : tree_fwd_spline_kernel<kFwdPose>;
  const cudaError_t e = allow_smem((const void*)kern, smem);
  if (e != cudaSuccess) return e;
  fit_carveout((const void*)kern, threads, smem);
  const int64_t grid = (a.B + threads - 1) / threads;
  kern<<<(unsigned)grid, threads, smem, s>>>(r, wt, a, sp);
  return cudaGetLastError();
}

cudaError_t launch_tree_bwd_spline_cost(const DevRobot& r, const WalkTab& wt, const BwdArgs& a,
                                        const FusedCost& fc, const SplineArgs& sp, int threads,
                                        int segments, cudaStream_t s) {
  if (threads <= 0) threads = 128;
  const int opt = bwd_opt(r, a, false);
  const int CG = segments > 1 ? seg_groups(segments, threads) : threads / 32;
  const int block = 32 * segments * CG;
  const size_t smem = (segments > 1 ? tree_seg_smem(r, segments, threads, false, true)
                                    : rec_smem(r, false)) +
                      12 * sizeof(float) * block +
                      (a.g_pose || a.g_sph ? grad_slot_smem(segments, threads) : 0);
  if (segments > 1)
    return launch_bwd(opt == 0            ? tree_bwd_spline_cost_seg_kernel<0>
                      : opt == kBwdSphere ? tree_bwd_spline_cost_seg_kernel<kBwdSphere>
                                          : tree_bwd_spline_cost_seg_kernel<kBwdGeneral>,
                      a.B, CG, block, smem, s, r, wt, a, fc, sp, seg_plan(segments));
  return launch_bwd(opt == 0            ? tree_bwd_spline_cost_kernel<0>
                    : opt == kBwdSphere ? tree_bwd_spline_cost_kernel<kBwdSphere>
                                        : tree_bwd_spline_cost_kernel<kBwdGeneral>,
                    a.B, CG, block, smem, s, r, wt, a, fc, sp);
}

int tree_max_depth() { return TMAXD; }

}  // namespace wbe
