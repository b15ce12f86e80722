// Two D2Q9 cells at a time for the runs of updates on the moments
// (lbrr_run2.cu, lbrr_run2m.cu): collision, sums, and the layout of the moments
// in memory.
#pragma once

#include "lbrr_launch.h"
#include "lbrr_quot.cuh"

namespace lbrr {
namespace two {

// ------------------------------------------------------ two cells at a time --
// The collision of lbrr_device.cuh (RR on D2Q9) on float2 values, one packed
// FP32x2 instruction of the sm_100 family an operation: the operations of the
// single updates in their order, so the bits are theirs. (With the outer
// populations at twice their value inside the chip, which leaves factors of 1/2
// out, a value that underflows was rounded elsewhere; 3% faster.)
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

// minus_reciprocal of both
__device__ __forceinline__ V minus_reciprocals(V x) {
  const V r = make_float2(approx_reciprocal(-x.x), approx_reciprocal(-x.y));
  return fma(fma(x, r, bc(1.0f)), r, r);
}
// u = j / rho correctly rounded: the quotient by the reciprocal of rho, corrected
// by its exact remainder (P. Markstein, IBM J. Res. Dev. 34, 1990; taken as
// rho q - j, with minus the reciprocal, so that a zero keeps its sign).
__device__ __forceinline__ Mac2 macro_of(const Mom2 &v) {
  Mac2 m;
  m.drho = v.drho;
  m.rho = add(bc(1.0f), m.drho);
  m.jx = v.jx;
  m.jy = v.jy;
  const V nx = muls(-1.0f, m.jx), ny = muls(-1.0f, m.jy);
  const V nr = minus_reciprocals(m.rho);
  const V qx = mul(nx, nr), qy = mul(ny, nr);
  m.ux = fma(fma(m.rho, qx, nx), nr, qx);
  m.uy = fma(fma(m.rho, qy, ny), nr, qy);
  const float least =
      fminf(fminf(fabsf(m.ux.x), fabsf(m.ux.y)), fminf(fabsf(m.uy.x), fabsf(m.uy.y)));
  if (!(least >= kLeastQuotient)) {
    if (needs_division(m.jx.x, m.ux.x) || needs_division(m.jx.y, m.ux.y) ||
        needs_division(m.jy.x, m.uy.x) || needs_division(m.jy.y, m.uy.y)) {
      m.ux = make_float2(__fdiv_rn(m.jx.x, m.rho.x), __fdiv_rn(m.jx.y, m.rho.y));
      m.uy = make_float2(__fdiv_rn(m.jy.x, m.rho.x), __fdiv_rn(m.jy.y, m.rho.y));
    }
  }
  m.pxx = fma(nx, m.ux, fmas(-kCs2, m.drho, v.xx));
  m.pxy = fma(nx, m.uy, v.xy);
  m.pyy = fma(ny, m.uy, fmas(-kCs2, m.drho, v.yy));
  return m;
}

// mom3 of lbrr_device.cuh
__device__ __forceinline__ void sum3(V a, V b, V c, V &s0, V &s1, V &s2) {
  s2 = add(a, c);
  s0 = add(s2, b);
  s1 = sub(c, a);
}
__device__ __forceinline__ Mom2 moments_of(const V (&f)[9]) {
  V s0[3], s1[3], s2[3], t0, t1, t2;
#pragma unroll
  for (int l = 0; l < 3; ++l) sum3(f[3 * l], f[3 * l + 1], f[3 * l + 2], s0[l], s1[l], s2[l]);
  Mom2 m;
  sum3(s0[0], s0[1], s0[2], m.drho, m.jy, m.yy);
  sum3(s1[0], s1[1], s1[2], m.jx, m.xy, t0);
  sum3(s2[0], s2[1], s2[2], m.xx, t1, t2);
  return m;
}

// The outer two populations come out as twice their value. TWICE: so do the
// coefficients come in; the factor 1/2 of coefficient 1 goes into the two sums it
// enters, as the compiler has it in the single updates, and the others take it by
// themselves, so that a value which underflows is rounded where theirs is.
template <bool TWICE>
__device__ __forceinline__ void synth3(V c0, V c1, V c2, V &om, V &oz, V &op) {
  if (TWICE) c0 = muls(0.5f, c0), c2 = muls(0.5f, c2);
  const V q = fmas(kCs2, c0, c2);
  oz = sub(c0, q);
  op = TWICE ? fmas(0.5f, c1, q) : add(q, c1);
  om = TWICE ? fmas(-0.5f, c1, q) : sub(q, c1);
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
  for (int b = 0; b < 3; ++b)
    synth3<false>(c[0][b], c[1][b], c[2][b], s[0][b], s[1][b], s[2][b]);
  synth3<true>(s[0][0], s[0][1], s[0][2], f[0], f[3], f[6]);
  synth3<false>(s[1][0], s[1][1], s[1][2], f[1], f[4], f[7]);
  synth3<true>(s[2][0], s[2][1], s[2][2], f[2], f[5], f[8]);
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    f[i] = muls(0.5f, f[i]);
    f[i + 6] = muls(0.5f, f[i + 6]);
  }
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
