// green.cuh -- the k-space multiply of the z passes (colpass.cuh, yz_kernels.cuh).
//
// At wave vector p (q = p except 0 in a Nyquist component):
//   X <- [X + q (q.X) f] d,  f = 1 / (|p|^2 - |q|^2 - kt2),  d = 1 / (N (|p|^2 - kt2)),
// the inverse of |p|^2 I - q q^T - kt2 I over N, kt2 = k0^2 + i epsilon.  A Nyquist component (even
// axis length, wave number pi/pitch whose sign is undefined) is 0 in q, which keeps the discrete
// curl curl real and symmetric; away from Nyquist this is (I - p p^T / kt2) / (|p|^2 - kt2), the
// dyadic Green's function of curl curl - kt2 (the vector CBS of refs. [25], [26] of arXiv 2506.15411).
//
// The same f and d act in every iteration, so their errors add up over a series where those of
// the field's values mostly do not.  Hence: |p|^2 - |q|^2 is built by selection (p p - q q leaves,
// contracted, the rounding error of p p, up to 5e-7 against |kt2| of 0.15 to 1); the tables hold
// squares rounded once from FP64; kt2 leaves |p|^2 before the square of pz is added; and d, whose
// reciprocal is the fast one, is corrected by its own residual, in which the part of 1/N beyond
// FP32 is made good too: five instructions more a mode.  With the constants of fft_radix.cuh and the
// phased twiddles of axis_plan.h, geometric means of the errors against 64 bits over 316 solves of
// 0.03 to 2.5 million voxels, before -> now: field 0.99 -> 0.57e-6, adjoint field 1.74 -> 0.97e-6, gradient
// 2.10 -> 1.20e-6 (staged passes on every axis: 1.00, 1.79, 2.23e-6).
#pragma once
#include "fft_radix.cuh"

namespace cbs {

// 1 / (re - i e), its reciprocal corrected once.
__device__ __forceinline__ float2 green_recip(float re, float e) {
  const float r = __fdividef(1.0f, fmaf(re, re, e * e));
  const float x = re * r, y = e * r;
  const float t = fmaf(-e, y, fmaf(-re, x, 1.0f));
  return make_float2(fmaf(x, t, x), fmaf(y, t, y));
}

// What the modes of one (x, y) column share.
struct GreenColumn {
  float qx, qy;
  float p2;     // px^2 + py^2 - Re kt2
  float nyq2;   // squares of its Nyquist components
  float2 f;     // f where pz is not Nyquist
};

// a + b as s + lo
__device__ __forceinline__ float two_sum(float a, float b, float& lo) {
  const float s = __fadd_rn(a, b), t = __fadd_rn(s, -a);
  lo = __fadd_rn(__fadd_rn(a, -__fadd_rn(s, -t)), __fadd_rn(b, -t));
  return s;
}

// px, py: (p^2, q) of the column's x and y frequencies.
__device__ __forceinline__ GreenColumn green_column(float2 px, float2 py, float2 kt2) {
  GreenColumn g;
  g.qx = px.y;
  g.qy = py.y;
  float l0, l1;
  const float s = two_sum(py.x, -kt2.x, l0);
  const float u = two_sum(px.x, s, l1);
  g.p2 = __fadd_rn(u, __fadd_rn(l0, l1));
  g.nyq2 = (px.y == 0.f ? px.x : 0.f) + (py.y == 0.f ? py.x : 0.f);   // (p = 0 adds nothing)
  g.f = green_recip(g.nyq2 - kt2.x, kt2.y);
  return g;
}

// pz: (p^2, q) of the z frequency; invN + invN rest: 1 / N.
__device__ __forceinline__ void green(const GreenColumn& g, float2 pz, float2 kt2, float invN, float rest, float2& X0,
                                      float2& X1, float2& X2) {
  float2 f = g.f;
  if (pz.y == 0.f && pz.x != 0.f) f = green_recip(g.nyq2 + pz.x - kt2.x, kt2.y);
  const float2 qd = cfma_r(pz.y, X2, cfma_r(g.qy, X1, make_float2(g.qx * X0.x, g.qx * X0.y)));
  const float2 c = cmul(qd, f);
  const float re = g.p2 + pz.x, e = kt2.y;
  const float r = __fdividef(1.0f, fmaf(re, re, e * e));
  const float x = re * r, y = e * r;
  const float t = (fmaf(-e, y, fmaf(-re, x, 1.0f)) + rest) * invN;
  const float2 d = make_float2(fmaf(x, invN, x * t), fmaf(y, invN, y * t));
  X0 = cmul(cfma_r(g.qx, c, X0), d);
  X1 = cmul(cfma_r(g.qy, c, X1), d);
  X2 = cmul(cfma_r(pz.y, c, X2), d);
}

}  // namespace cbs
