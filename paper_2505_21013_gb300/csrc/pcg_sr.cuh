// Arithmetic of the single-reduction PCG, shared by its kernels (pcg_sr.cu, pcg_su.cu).
#pragma once

#include "pcg_common.cuh"

namespace ppn {
namespace pcgdev {

// ---- the arithmetic every layout shares (explicit rounding, so that all kernels and
// layouts, and a halo row and its owner, give the same bits)
// a BSR block times v, accumulated: ax += a[0:3].v, ay += a[3:6].v, az += a[6:9].v
__device__ __forceinline__ void blk_mv(const float* a, float vx, float vy, float vz, float& ax, float& ay,
                                       float& az) {
  ax = __fmaf_rn(a[2], vz, __fmaf_rn(a[1], vy, __fmaf_rn(a[0], vx, ax)));
  ay = __fmaf_rn(a[5], vz, __fmaf_rn(a[4], vy, __fmaf_rn(a[3], vx, ay)));
  az = __fmaf_rn(a[8], vz, __fmaf_rn(a[7], vy, __fmaf_rn(a[6], vx, az)));
}
__device__ __forceinline__ float dot3(float a0, float a1, float a2, float b0, float b1, float b2) {
  return __fmaf_rn(a2, b2, __fmaf_rn(a1, b1, __fmul_rn(a0, b0)));
}
// u = P r, P symmetric, q = its entries 00 01 02 11 12 22
__device__ __forceinline__ void prec6(const float* q, const float* r, float* u) {
  u[0] = dot3(q[0], q[1], q[2], r[0], r[1], r[2]);
  u[1] = dot3(q[1], q[3], q[4], r[0], r[1], r[2]);
  u[2] = dot3(q[2], q[4], q[5], r[0], r[1], r[2]);
}
__device__ __forceinline__ void sym6(const float* P, float* q) {
  q[0] = P[0], q[1] = P[1], q[2] = P[2], q[3] = P[4], q[4] = P[5], q[5] = P[8];
}
// s = w + beta s, r -= alpha s (one component): the part a halo row repeats
__device__ __forceinline__ void upd_sr(float a, float b, float w, float& sv, float& r) {
  sv = __fmaf_rn(b, sv, w);
  r = __fmaf_rn(-a, sv, r);
}
// p = u + beta p, x += alpha p (one component)
__device__ __forceinline__ void upd_px(float a, float b, float u, float& p, float& x) {
  p = __fmaf_rn(b, p, u);
  x = __fmaf_rn(a, p, x);
}
__device__ __forceinline__ void st_relaxed_v2_u64(unsigned long long* p, unsigned long long a, unsigned long long b) {
  asm volatile("st.relaxed.gpu.global.v2.u64 [%0], {%1,%2};" ::"l"(p), "l"(a), "l"(b) : "memory");
}
__device__ __forceinline__ void ld_relaxed_v2_u64(const unsigned long long* p, unsigned long long& a,
                                                  unsigned long long& b) {
  asm volatile("ld.relaxed.gpu.global.v2.u64 {%0,%1}, [%2];" : "=l"(a), "=l"(b) : "l"(p) : "memory");
}

// scalar step after the reduction of iteration `it` (it updates done so far):
// stopping tests, then alpha and beta of the next direction, or the exits
__device__ __forceinline__ void sr_step(SState<float>& s, float gam, float del, float rho, float fail, int it,
                                        float tol2, int max_iter) {
  s.rr = rho;
  if (it == 0) {
    s.rr0 = rho;
    s.pfail = fail > 0.0f;
    s.ind = fail > 0.0f;
    s.iters = 0;
    s.hitmax = 0;
    s.nonfinite = !(rho == rho) || !(gam == gam);
    if (s.ind || s.nonfinite || !(rho > 0.0f)) {
      s.done = 1;
      return;
    }
  }
  if (!(rho == rho) || !(gam == gam) || !(del == del)) {
    s.nonfinite = 1;
    s.done = 1;
    return;
  }
  if (it > 0 && rho <= tol2 * s.rr0) {
    s.done = 1;
    return;
  }
  if (it > 0 && s.iters >= max_iter) {
    s.hitmax = 1;
    s.done = 1;
    return;
  }
  const float beta = it > 0 ? gam / s.rz : 0.0f;
  const float d = it > 0 ? del - beta * gam / s.alpha : del;  // p^T A p of the next direction
  s.dq = d;
  if (!(d > 0.0f)) {
    if (!(d == d)) s.nonfinite = 1;
    s.ind = 1;
    s.done = 1;
    return;
  }
  s.beta = beta;
  s.alpha = gam / d;
  s.rz = gam;
}

}  // namespace pcgdev
}  // namespace ppn
