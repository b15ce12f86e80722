// Two D2Q9 cells at a time for the runs of updates on the moments
// (lbrr_run2.cu, lbrr_run2m.cu): collision, sums, and the layout of the moments
// in memory.
#pragma once

#include "lbrr_launch.h"

namespace lbrr {
namespace two {

// ------------------------------------------------------ two cells at a time --
// The collision of lbrr_device.cuh (RR on D2Q9) on float2 values, one packed
// FP32x2 instruction of the sm_100 family an operation: the operations of the
// single updates in their order, so the bits are theirs.
using V = float2;
__device__ __forceinline__ V bc(float s) { return make_float2(s, s); }
__device__ __forceinline__ V add(V a, V b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ V mul(V a, V b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ V fma(V a, V b, V c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ V sub(V a, V b) { return __ffma2_rn(b, bc(-1.0f), a); }  // one rounding
__device__ __forceinline__ V muls(float s, V b) { return __fmul2_rn(bc(s), b); }
__device__ __forceinline__ V fmas(float s, V b, V c) { return __ffma2_rn(bc(s), b, c); }

// What a cell carries from update to update: rho - 1, rho u and its raw second
// moments.
struct Mom2 {
  V drho, jx, jy, xx, xy, yy;
};
struct Mac2 {
  V drho, rho, jx, jy, ux, uy, pxx, pxy, pyy;
};

// j / rho correctly rounded (P. Markstein, IBM J. Res. Dev. 34, 1990): one
// Newton step takes the 1-ulp approximation to the correctly rounded
// reciprocal, one correction by the exact remainder the quotient to its own.
__device__ __forceinline__ float rcp_approx(float x) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
__device__ __forceinline__ void set_velocity(Mac2 &m) {
  m.rho = add(bc(1.0f), m.drho);
  const V nr = muls(-1.0f, m.rho);
  V r = make_float2(rcp_approx(m.rho.x), rcp_approx(m.rho.y));
  r = fma(fma(nr, r, bc(1.0f)), r, r);
  const V qx = mul(m.jx, r), qy = mul(m.jy, r);
  m.ux = fma(fma(nr, qx, m.jx), r, qx);
  m.uy = fma(fma(nr, qy, m.jy), r, qy);
}
__device__ __forceinline__ Mac2 macro_of(const Mom2 &v) {
  Mac2 m;
  m.drho = v.drho;
  m.jx = v.jx;
  m.jy = v.jy;
  set_velocity(m);
  const V nx = muls(-1.0f, m.jx);
  m.pxx = fma(nx, m.ux, fmas(-kCs2, m.drho, v.xx));
  m.pxy = fma(nx, m.uy, v.xy);
  m.pyy = fma(muls(-1.0f, m.jy), m.uy, fmas(-kCs2, m.drho, v.yy));
  return m;
}

// Populations inside the chip: f_i times 2^(number of its non-zero velocity
// components), which leaves the factors 1/2 out of the synthesis; the sums
// put them back (powers of two change no rounding short of underflow).
__device__ __forceinline__ void sum3(V a, V b, V c, V &s0, V &s1, V &s2) {
  s2 = add(a, c);
  s0 = fmas(0.5f, s2, b);
  s1 = sub(c, a);
}
__device__ __forceinline__ Mom2 moments_of(const V (&f)[9]) {
  V s0[3], s1[3], s2[3], t0, t1, t2;
#pragma unroll
  for (int l = 0; l < 3; ++l) sum3(f[3 * l], f[3 * l + 1], f[3 * l + 2], s0[l], s1[l], s2[l]);
  V m01, m02, m10, m11, m20;
  Mom2 m;
  sum3(s0[0], s0[1], s0[2], m.drho, m01, m02);
  sum3(s1[0], s1[1], s1[2], m10, m11, t0);
  sum3(s2[0], s2[1], s2[2], m20, t1, t2);
  m.jx = muls(0.5f, m10);
  m.jy = muls(0.5f, m01);
  m.xx = muls(0.5f, m20);
  m.xy = muls(0.25f, m11);
  m.yy = muls(0.5f, m02);
  return m;
}

__device__ __forceinline__ void synth3(V c0, V c1, V c2, V &om, V &oz, V &op) {
  const V q = fmas(kCs2, c0, c2);
  oz = sub(c0, q);
  op = add(q, c1);
  om = sub(q, c1);
}
__device__ __forceinline__ void post_collision(const Mac2 &m, float om1, V (&f)[9]) {
  const V uy = m.uy, uyy = mul(uy, uy), uxx = mul(m.ux, m.ux), ux2 = add(m.ux, m.ux);
  const V pxx = muls(om1, m.pxx), pyy = muls(om1, m.pyy), pxy = muls(om1, m.pxy);
  const V q1_1 = mul(m.rho, uy), q1_2 = fma(m.rho, uyy, pyy);
  const V q3_2 = mul(add(pxy, pxy), uy);
  V c[3][3], s[3][3];
  c[0][0] = m.drho;
  c[0][1] = m.jy;
  c[0][2] = q1_2;
  c[1][0] = m.jx;
  c[1][1] = fma(m.ux, q1_1, pxy);
  c[1][2] = fma(m.ux, q1_2, q3_2);
  c[2][0] = fma(uxx, m.rho, pxx);
  c[2][1] = fma(uxx, q1_1, fma(ux2, pxy, mul(pxx, uy)));
  c[2][2] = fma(uxx, q1_2, fma(ux2, q3_2, mul(pxx, uyy)));
#pragma unroll
  for (int b = 0; b < 3; ++b) synth3(c[0][b], c[1][b], c[2][b], s[0][b], s[1][b], s[2][b]);
#pragma unroll
  for (int ix = 0; ix < 3; ++ix) synth3(s[ix][0], s[ix][1], s[ix][2], f[ix], f[ix + 3], f[ix + 6]);
}

__host__ __device__ constexpr float scale2(int i) {
  return (vel(i, 0) ? 2.0f : 1.0f) * (vel(i, 1) ? 2.0f : 1.0f);
}
__device__ __forceinline__ float &lane(V &v, int k) { return k ? v.y : v.x; }

// ------------------------------------------------------------------ memory --
// Moments in memory: rows in blocks of 32 cells; of a block first rho - 1,
// rho u_x, rho u_y, Pi_xx of its cells as float4, then Pi_xy and Pi_yy as float2.
__host__ __device__ __forceinline__ int blocks2_x(const Grid &g) { return (g.nx + 31) / 32; }
__device__ __forceinline__ long long block2(const Grid &g, int x, int y) {
  return ((long long)y * blocks2_x(g) + (x >> 5)) * 192;
}

}  // namespace two
}  // namespace lbrr
