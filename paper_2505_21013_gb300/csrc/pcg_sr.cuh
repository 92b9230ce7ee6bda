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

// sr_step on the common path (another iteration follows) with its divisions issued at once, not
// behind one exit test after the other; the tests decide as sr_step does
__device__ __forceinline__ void sr_step_fast(SState<float>& s, float gam, float del, float rho, float fail, int it,
                                             float tol2, int max_iter) {
  const float rz = s.rz, alpha = s.alpha, rr0 = s.rr0;
  const int iters = s.iters;
  const float beta = gam / rz, d = del - beta * gam / alpha, a = gam / d;
  if (it > 0 && rho == rho && gam == gam && del == del && !(rho <= tol2 * rr0) && iters < max_iter && d > 0.0f) {
    s.rr = rho;
    s.dq = d;
    s.beta = beta;
    s.alpha = a;
    s.rz = gam;
  } else {
    sr_step(s, gam, del, rho, fail, it, tol2, max_iter);
  }
}

// ---- 16-byte words: three FP32 values and the 32-bit stamp, read and written as one 128-bit
// scalar (single-copy atomic): a word with the expected stamp carries its values
__device__ __forceinline__ void st_word4(float4* p, float x, float y, float z, unsigned s) {
  asm volatile(
      "{\n\t.reg .b128 w;\n\tmov.b128 w, {%1, %2};\n\tst.relaxed.gpu.global.b128 [%0], w;\n\t}" ::"l"(p),
      "l"(((unsigned long long)__float_as_uint(y) << 32) | __float_as_uint(x)),
      "l"(((unsigned long long)s << 32) | __float_as_uint(z))
      : "memory");
}
__device__ __forceinline__ void ld_word4(const float4* p, unsigned long long& a, unsigned long long& b) {
  asm volatile("{\n\t.reg .b128 w;\n\tld.relaxed.gpu.global.b128 w, [%2];\n\tmov.b128 {%0, %1}, w;\n\t}"
               : "=l"(a), "=l"(b)
               : "l"(p)
               : "memory");
}
__device__ __forceinline__ unsigned word4_stamp(unsigned long long b) { return (unsigned)(b >> 32); }

}  // namespace pcgdev
}  // namespace ppn
