// spatial.cuh -- compact spatial algebra on the device (Sec. 6.3, "Compact
// spatial representations", Tab. rnea_comparison).
//
// A link transform is a rotation R (row-major 3x3, child axes in parent
// coordinates) and a translation p (child origin in parent coordinates): 12
// floats instead of a 6x6 Plucker matrix.  Spatial vectors are [angular;
// linear] about the frame origin.
//   motion, parent -> child:  X m = [R^T w ; R^T (u + w x p)]
//   force,  child -> parent:  X^T f = [R n + p x (R f) ; R f]
// A spatial inertia is 10 floats (m, h = m c, Io = inertia about the link
// origin): I v = [Io w + h x u ; m u - h x w].
#pragma once

#include "wbe_internal.h"

#include <cuda_fp16.h>

namespace wbe {

__device__ __forceinline__ void cross3(const float* a, const float* b, float* c) {
  c[0] = fmaf(a[1], b[2], -a[2] * b[1]);
  c[1] = fmaf(a[2], b[0], -a[0] * b[2]);
  c[2] = fmaf(a[0], b[1], -a[1] * b[0]);
}

__device__ __forceinline__ float dot3(const float* a, const float* b) {
  return fmaf(a[2], b[2], fmaf(a[1], b[1], a[0] * b[0]));
}

// y = R x
__device__ __forceinline__ void rot(const float* R, const float* x, float* y) {
  y[0] = fmaf(R[2], x[2], fmaf(R[1], x[1], R[0] * x[0]));
  y[1] = fmaf(R[5], x[2], fmaf(R[4], x[1], R[3] * x[0]));
  y[2] = fmaf(R[8], x[2], fmaf(R[7], x[1], R[6] * x[0]));
}

// y = R^T x
__device__ __forceinline__ void rotT(const float* R, const float* x, float* y) {
  y[0] = fmaf(R[6], x[2], fmaf(R[3], x[1], R[0] * x[0]));
  y[1] = fmaf(R[7], x[2], fmaf(R[4], x[1], R[1] * x[0]));
  y[2] = fmaf(R[8], x[2], fmaf(R[5], x[1], R[2] * x[0]));
}

// C = A B (3x3 row-major)
__device__ __forceinline__ void matmul3(const float* A, const float* B, float* C) {
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j)
      C[3 * i + j] = fmaf(A[3 * i + 2], B[6 + j], fmaf(A[3 * i + 1], B[3 + j], A[3 * i] * B[j]));
}

// Robot parameters (fixed transforms, axes, mimic factors, inertias) are read
// with plain loads, not __ldg: the segmented backward sweeps stage them in
// shared memory and hand the sweep pointers into it.
template <class T>
__device__ __forceinline__ T ldp(const T* p) {
  return *p;
}

__device__ __forceinline__ float joint_var(const DevRobot& r, int k, float qj) {
  const float2 mm = reinterpret_cast<const float2*>(r.mimic)[k];
  return fmaf(mm.x, qj, mm.y);
}

// sin and cos of a joint angle: Cody and Waite's reduction (1980) of th to
// x = th - k 2 pi, k = rint(th / 2 pi), with 2 pi split as 6.28125 (8
// significant bits, so k * 6.28125 and th - k * 6.28125 are exact for
// |k| < 2^16) plus 1.93530718e-3 (the split's residual is 1.03e-11 per
// multiple of 2 pi), then CUDA's fast intrinsic on x in [-pi, pi], where
// its absolute error is at most 2^-21.41.  Overall within about 5e-7 of the
// exact sine and cosine of the float angle for |th| <= 4e4 rad (tested
// against double precision), a few times the rounding of a float sine; the
// sweeps evaluate it at every push and close, where the library sincosf's
// longer dependency chain cost 3 % (forward) and 5 % (backward) of the
// humanoid's sweep time.
__device__ __forceinline__ void joint_sincos(float th, float* s, float* c) {
  const float k = rintf(th * 0.159154943f);
  float x = fmaf(-k, 6.28125f, th);
  x = fmaf(-k, 1.93530718e-3f, x);
  __sincosf(x, s, c);
}

// Local transform of link k (parent joint frame -> link frame) for joint
// variable th: T_fixed * J(th).  Revolute: R = R_f R_J(th) with Rodrigues'
// rotation R_J = c I + s [a]^ + (1-c) a a^T.  Prismatic: p = p_f + R_f a th.
// (T4: T_fixed as three float4, a: the axis, jt, ident: the joint type and
// whether the fixed rotation is the identity; UNIT: the sine and cosine
// scaled to s^2 + c^2 = 1 within a rounding -- the fast pair misses it by up to
// 7e-7 -- so that R's inverse is its transpose and products of many R stay
// rotations)
template <bool UNIT = false>
__device__ __forceinline__ void local_xf_q(const float4* T4, float4 a, float th, int jt,
                                           bool ident, float* R, float* p) {
  const float4 t2 = T4[2];
  p[0] = t2.y;
  p[1] = t2.z;
  p[2] = t2.w;
  if (jt == 1) {
    float s, c;
    joint_sincos(th, &s, &c);
    if (UNIT) {
      const float u = 0.5f * fmaf(-s, s, fmaf(-c, c, 1.0f));
      s = fmaf(s, u, s);
      c = fmaf(c, u, c);
    }
    const float t = 1.0f - c;
    const float tx = t * a.x, ty = t * a.y, tz = t * a.z;
    const float sx = s * a.x, sy = s * a.y, sz = s * a.z;
    float Rj[9];
    Rj[0] = fmaf(tx, a.x, c);
    Rj[1] = fmaf(tx, a.y, -sz);
    Rj[2] = fmaf(tx, a.z, sy);
    Rj[3] = fmaf(ty, a.x, sz);
    Rj[4] = fmaf(ty, a.y, c);
    Rj[5] = fmaf(ty, a.z, -sx);
    Rj[6] = fmaf(tz, a.x, -sy);
    Rj[7] = fmaf(tz, a.y, sx);
    Rj[8] = fmaf(tz, a.z, c);
    if (ident) {
#pragma unroll
      for (int i = 0; i < 9; ++i) R[i] = Rj[i];
    } else {
      const float4 t0 = T4[0], t1 = T4[1];
      const float Rf[9] = {t0.x, t0.y, t0.z, t0.w, t1.x, t1.y, t1.z, t1.w, t2.x};
      matmul3(Rf, Rj, R);
    }
  } else {
    const float4 t0 = T4[0], t1 = T4[1];
    const float Rf[9] = {t0.x, t0.y, t0.z, t0.w, t1.x, t1.y, t1.z, t1.w, t2.x};
#pragma unroll
    for (int i = 0; i < 9; ++i) R[i] = Rf[i];
    if (jt == 2) {
      const float s[3] = {a.x * th, a.y * th, a.z * th};
      float Rs[3];
      rot(Rf, s, Rs);
      p[0] += Rs[0];
      p[1] += Rs[1];
      p[2] += Rs[2];
    }
  }
}

__device__ __forceinline__ void local_xf(const DevRobot& r, int k, float th, float* R, float* p) {
  local_xf_q(reinterpret_cast<const float4*>(r.Tf + 12 * k),
             reinterpret_cast<const float4*>(r.axis)[k], th, __ldg(r.jtype + k),
             __ldg(r.rot_id + k) != 0, R, p);
}

// motion vector m (parent coords) -> child coords
__device__ __forceinline__ void xf_motion(const float* R, const float* p, const float* m,
                                          float* out) {
  float wxp[3], t[3];
  cross3(m, p, wxp);
  t[0] = m[3] + wxp[0];
  t[1] = m[4] + wxp[1];
  t[2] = m[5] + wxp[2];
  rotT(R, m, out);
  rotT(R, t, out + 3);
}

// force vector f (child coords) -> parent coords (X^T f); the same map
// carries adjoints of motion vectors back to the parent.
__device__ __forceinline__ void xf_force_T(const float* R, const float* p, const float* f,
                                           float* out) {
  float Rn[3], pxRf[3];
  rot(R, f + 3, out + 3);
  rot(R, f, Rn);
  cross3(p, out + 3, pxRf);
  out[0] = Rn[0] + pxRf[0];
  out[1] = Rn[1] + pxRf[1];
  out[2] = Rn[2] + pxRf[2];
}

// crm(v) m = [w x mw ; u x mw + w x mu]
__device__ __forceinline__ void crm(const float* v, const float* m, float* out) {
  float a[3], b[3];
  cross3(v, m, out);
  cross3(v + 3, m, a);
  cross3(v, m + 3, b);
  out[3] = a[0] + b[0];
  out[4] = a[1] + b[1];
  out[5] = a[2] + b[2];
}

// crf(v) f = [w x fn + u x ff ; w x ff]
__device__ __forceinline__ void crf(const float* v, const float* f, float* out) {
  float a[3], b[3];
  cross3(v, f, a);
  cross3(v + 3, f + 3, b);
  out[0] = a[0] + b[0];
  out[1] = a[1] + b[1];
  out[2] = a[2] + b[2];
  cross3(v, f + 3, out + 3);
}

// I v for the compact inertia {m, h[3], Io[6] = xx yy zz xy xz yz}
__device__ __forceinline__ void inertia_mul(const float* I, const float* v, float* out) {
  const float m = I[0];
  const float h[3] = {I[1], I[2], I[3]};
  const float* w = v;
  const float* u = v + 3;
  float hxu[3], hxw[3];
  cross3(h, u, hxu);
  cross3(h, w, hxw);
  out[0] = fmaf(I[4], w[0], fmaf(I[7], w[1], fmaf(I[8], w[2], hxu[0])));
  out[1] = fmaf(I[7], w[0], fmaf(I[5], w[1], fmaf(I[9], w[2], hxu[1])));
  out[2] = fmaf(I[8], w[0], fmaf(I[9], w[1], fmaf(I[6], w[2], hxu[2])));
  out[3] = fmaf(m, u[0], -hxw[0]);
  out[4] = fmaf(m, u[1], -hxw[1]);
  out[5] = fmaf(m, u[2], -hxw[2]);
}

__device__ __forceinline__ void load_inertia(const DevRobot& r, int k, float* I) {
  const float* src = r.inert + 10 * k;
#pragma unroll
  for (int i = 0; i < 10; ++i) I[i] = ldp(src + i);
}

// Joint motion subspace S of link k as (jt, axis): revolute [a;0],
// prismatic [0;a], fixed 0.  Helpers for S^T x and S * s.
__device__ __forceinline__ float St_dot(int jt, const float* a, const float* x) {
  return jt == 1 ? dot3(a, x) : (jt == 2 ? dot3(a, x + 3) : 0.0f);
}

// RNEA forward sweep for one link (Alg. 4, pass 1): given the parent's
// velocity/acceleration (parent coords), the local transform and the joint
// rates, produce v_k and a_k in link coordinates:
//   v = X v_pa + S qd ;  a = X a_pa + S qdd + v x_m (S qd)
__device__ __forceinline__ void rnea_va(const float* R, const float* p, const float* vpa,
                                        const float* apa, int jt, const float* ax, float qd,
                                        float qdd, float* v, float* a) {
  xf_motion(R, p, vpa, v);
  xf_motion(R, p, apa, a);
  if (jt == 1) {
    const float s[3] = {ax[0] * qd, ax[1] * qd, ax[2] * qd};
    v[0] += s[0];
    v[1] += s[1];
    v[2] += s[2];
    float wxs[3], uxs[3];
    cross3(v, s, wxs);
    cross3(v + 3, s, uxs);
    a[0] += fmaf(ax[0], qdd, wxs[0]);
    a[1] += fmaf(ax[1], qdd, wxs[1]);
    a[2] += fmaf(ax[2], qdd, wxs[2]);
    a[3] += uxs[0];
    a[4] += uxs[1];
    a[5] += uxs[2];
  } else if (jt == 2) {
    const float s[3] = {ax[0] * qd, ax[1] * qd, ax[2] * qd};
    v[3] += s[0];
    v[4] += s[1];
    v[5] += s[2];
    float wxs[3];
    cross3(v, s, wxs);
    a[3] += fmaf(ax[0], qdd, wxs[0]);
    a[4] += fmaf(ax[1], qdd, wxs[1]);
    a[5] += fmaf(ax[2], qdd, wxs[2]);
  }
}

// Alg. 4, pass 2: f = I a + v x* (I v)
__device__ __forceinline__ void rnea_force(const float* I, const float* v, const float* a,
                                           float* f) {
  float Ia[6], Iv[6], c[6];
  inertia_mul(I, a, Ia);
  inertia_mul(I, v, Iv);
  crf(v, Iv, c);
#pragma unroll
  for (int i = 0; i < 6; ++i) f[i] = Ia[i] + c[i];
}

// Squared centre distance with a fixed operation order, shared by the fast
// filter and the exact path of the pair stage.
__device__ __forceinline__ float dist2(float xi, float yi, float zi, float xj, float yj,
                                       float zj) {
  const float dx = xi - xj, dy = yi - yj, dz = zi - zj;
  return fmaf(dz, dz, fmaf(dy, dy, dx * dx));
}

// entry i of the schedule's arrays for the bounds (round_entry), as `ent` has it
__device__ __forceinline__ uint2 sched_at(const PairSchedule32& ps, int i) {
  return make_uint2(__ldg(reinterpret_cast<const uint32_t*>(ps.off) + i) << 1,
                    __ldg(reinterpret_cast<const uint32_t*>(ps.blk) + i));
}

// approximate square root (relative error at most 2^-23)
__device__ __forceinline__ float sqrt_approx(float x) {
  float y;
  asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// A bounding sphere of a group of collision spheres as four halves (x, y and
// z, radius): the centre rounded, the radius grown by what that moved it and by
// 5e-4 (the rounding of a sum of two radii), rounded up -- still a bound.  The
// pair stage reads two of them for every block of every configuration, and the
// shared memory's wavefronts, half as many for 8 bytes, are what it runs out of.
// A coordinate beyond 32752 makes the radius infinite: two such could differ by
// more than a half holds, and their gap would come out as infinite.
__device__ __forceinline__ uint2 half_bound(float x, float y, float z, float R) {
  const __half2 xy = __floats2half2_rn(x, y);
  const __half hz = __float2half_rn(z);
  const float2 f = __half22float2(xy);
  const float e = fabsf(x - f.x) + fabsf(y - f.y) + fabsf(z - __half2float(hz));
  const bool fits = fmaxf(fabsf(x), fmaxf(fabsf(y), fabsf(z))) <= 32752.0f;
  const float grown = fits ? (R + e) * 1.0005f : __int_as_float(0x7f800000);
  const __half2 zr = __halves2half2(hz, __float2half_ru(grown));
  return make_uint2(*reinterpret_cast<const uint32_t*>(&xy), *reinterpret_cast<const uint32_t*>(&zr));
}
// The bound of a group over several links: the mean of its m centres, and the
// farthest sphere's reach from it, widened by 1e-6 of itself (the approximate
// square root's error is 2^-23 of it) and of the centre's place, and by ow.
// X, Y, Z: the 4 centres (0 past the m-th), rad: their radii; ox, oy, oz: the
// origin the bound is relative to.
__device__ __forceinline__ uint2 mixed_bound(float4 X, float4 Y, float4 Z, float4 rad, int m,
                                             float ox, float oy, float oz, float ow) {
  const float inv = m >= 4 ? 0.25f : m == 3 ? 1.0f / 3.0f : m == 2 ? 0.5f : 1.0f;
  const float cx = (X.x + X.y + X.z + X.w) * inv, cy = (Y.x + Y.y + Y.z + Y.w) * inv,
              cz = (Z.x + Z.y + Z.z + Z.w) * inv;
  auto reach = [&](float x, float y, float z, float r) {
    return sqrt_approx(dist2(cx, cy, cz, x, y, z)) + r;
  };
  float R = m > 0 ? reach(X.x, Y.x, Z.x, rad.x) : 0.0f;
  if (m > 1) R = fmaxf(R, reach(X.y, Y.y, Z.y, rad.y));
  if (m > 2) R = fmaxf(R, reach(X.z, Y.z, Z.z, rad.z));
  if (m > 3) R = fmaxf(R, reach(X.w, Y.w, Z.w, rad.w));
  const float dx = cx - ox, dy = cy - oy, dz = cz - oz;
  const float e = fmaf(fabsf(dx) + fabsf(dy) + fabsf(dz), 1e-6f, ow);
  return half_bound(dx, dy, dz, fmaf(R, 1e-6f, R) + e);
}
// The sphere that stands for the groups of a null block: far from every finite
// bound, so that a null block is rarely kept (and then has no pair to work).
__device__ __forceinline__ uint2 far_bound() {
  const __half2 xy = __floats2half2_rn(6e4f, 6e4f), zr = __floats2half2_rn(6e4f, 0.0f);
  return make_uint2(*reinterpret_cast<const uint32_t*>(&xy), *reinterpret_cast<const uint32_t*>(&zr));
}
// Lower bound of the distance between the surfaces of two such spheres (and so
// of any spheres within them): differences in half are off by at most 2^-11 of
// themselves, which 6e-4 of the distance covers with the square root's error.
// Finite bounds' coordinates never overflow; where a radius or the sum of two
// does, the gap is minus infinity or not a number: a caller has to keep both.
__device__ __forceinline__ float half_gap(uint2 a, uint2 b) {
  const __half2 axy = *reinterpret_cast<const __half2*>(&a.x), azr = *reinterpret_cast<const __half2*>(&a.y);
  const __half2 bxy = *reinterpret_cast<const __half2*>(&b.x), bzr = *reinterpret_cast<const __half2*>(&b.y);
  const __half2 d = __hsub2(axy, bxy), zr = __hfma2(bzr, __floats2half2_rn(-1.0f, 1.0f), azr);
  float d2;  // squares of halves added in fp32
  asm("{\n\t.reg .f16 x, y, z, r;\n\t.reg .f32 s;\n\t"
      "mov.b32 {x, y}, %1;\n\tmov.b32 {z, r}, %2;\n\t"
      "fma.rn.f32.f16 s, x, x, 0f00000000;\n\tfma.rn.f32.f16 s, y, y, s;\n\t"
      "fma.rn.f32.f16 %0, z, z, s;\n\t}"
      : "=f"(d2)
      : "r"(*reinterpret_cast<const uint32_t*>(&d)), "r"(*reinterpret_cast<const uint32_t*>(&zr)));
  return fmaf(sqrt_approx(d2), 0.9994f, -__high2float(zr));
}

}  // namespace wbe
