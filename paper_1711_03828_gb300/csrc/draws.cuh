// draws.cuh -- what the smart Monte Carlo and learned moves make of their
// Philox draws: the accurate ln of an open uniform, the phase of a uniform
// angle, the acceptance uniform from a draw's spare bits, and the three
// Box-Muller normals of a move (internal; the uniform move's transforms are
// in common.cuh).
#pragma once

#include "common.cuh"

namespace soma {

// log1p(f) for the reduced argument f in [sqrt(1/2) - 1, sqrt(2) - 1] by the
// series log(1 + f) = 2 atanh(s) = 2 (s + s^3/3 + s^5/5 + ...), s = f/(2 + f),
// |s| <= 3 - 2 sqrt(2) < 0.1716: five terms leave a truncation below s^10/11 <
// 5e-9 relative, under the FP32 rounding of the terms; s is the correctly
// rounded quotient of f and the rounded 2 + f (about one ulp).  Near f = 0 the
// result keeps the relative accuracy of f itself.
__device__ __forceinline__ float log1p_reduced(float f) {
  const float s = __fdiv_rn(f, 2.f + f);
  const float z = s * s;
  float t = fmaf(z, 0.111111111111111111f, 0.142857142857142857f);   // 1/9, 1/7
  t = fmaf(z, t, 0.2f);
  t = fmaf(z, t, 0.333333333333333333f);
  const float ss = s + s;
  return fmaf(ss * z, t, ss);
}

// ln of the open uniform u = (k + 1/2)/2^24, accurate to about one FP32 ulp of
// the result for every k, without a branch on k (a warp's lanes fall on both
// sides of u = 1/2 at random).  Below 1/2, u itself is exact in FP32; above,
// v = 1 - u = (2^24 - k - 1/2)/2^24 is exact instead.  Either is reduced to
// ln u = e ln 2 + log1p(f) with f = m - 1 exact and m in [sqrt(1/2), sqrt(2))
// (Cody and Waite's argument reduction): u = 2^e m from the exponent bits
// below 1/2; above, m = u (e = 0, f = -v) for u >= sqrt(1/2) and m = 2u
// (e = -1, f = 1 - 2v) below it.  ln 2 enters split in a part whose products
// with e are exact and a small correction.
__device__ __forceinline__ float log_uniform_open_accurate(uint32_t r) {
  const uint32_t k = r >> 8;
  const bool upper = k >= (1u << 23);
  const float u = fmaf(__uint2float_rn(k), 5.9604644775390625e-8f, 2.98023223876953125e-8f);
  const float v = fmaf(__uint2float_rn((1u << 24) - k), 5.9604644775390625e-8f,
                       -2.98023223876953125e-8f);
  // lower half: u = 2^e m, m in [1, 2), then halved into [sqrt(1/2), sqrt(2))
  const uint32_t b = __float_as_uint(u);
  float m = __uint_as_float((b & 0x007FFFFFu) | 0x3F800000u);
  int e = (int)(b >> 23) - 127;
  const bool halve = m >= 1.41421356237309505f;
  m = halve ? 0.5f * m : m;
  e += halve ? 1 : 0;
  // upper half: e = 0 above sqrt(1/2), else -1
  const bool e0 = v <= 0.29289321881345248f;   // 1 - sqrt(1/2)
  const float f = upper ? (e0 ? -v : fmaf(-2.f, v, 1.f)) : m - 1.f;
  const float ef = (float)(upper ? (e0 ? 0 : -1) : e);
  return fmaf(ef, 0.693145751953125f, fmaf(ef, 1.428606820309417232e-6f, log1p_reduced(f)));
}

// The 24 bits of a move draw r that its four top-24-bit uniforms leave over
// (the low bytes of words x, y, z; x's lowest), as the top 24 bits of a word:
// the acceptance uniform of a move whose four uniforms are all taken.
__device__ __forceinline__ uint32_t spare_uniform_word(const uint4& r) {
  return ((r.x & 0xFFu) | (r.y & 0xFFu) << 8 | (r.z & 0xFFu) << 16) << 8;
}

// cos and sin of 2 pi u for the open uniform u = (k + 1/2)/2^24: with the exact
// symmetric uniform v = 2u - 1, 2 pi u = pi v + pi, so cos = -cospi(v) and
// sin = -sinpi(v), evaluated without rounding the phase.
__device__ __forceinline__ void sincos_2pi_uniform(uint32_t r, float* s, float* c) {
  float sv, cv;
  sincospif(uniform_sym(r), &sv, &cv);
  *s = -sv;
  *c = -cv;
}

// The same with the hardware approximations (__sincosf of the phase reduced
// to [-pi, pi)): absolute error about 2^-21, for proposals whose acceptance
// uses the realised trial position rather than the draw.
__device__ __forceinline__ void sincos_2pi_uniform_fast(uint32_t r, float* s, float* c) {
  const float u = fmaf(__uint2float_rn(r >> 8), 5.9604644775390625e-8f, 2.98023223876953125e-8f);
  __sincosf(fmaf(6.2831853071795865f, u, -3.1415926535897932f), s, c);
  *s = -*s;
  *c = -*c;
}

// sqrt(-2 ln u) of the open uniforms of two draw words at once, in packed FP32x2
// instructions: the values of sqrtf(-2.f * log_uniform_open_accurate(r)), bit for
// bit, in half the FP32 instructions.  The correctly rounded quotient and root
// come without the general functions' range checks: approximate reciprocal and
// reciprocal root, one Newton step, and the residual correction of Markstein
// (IBM J. Res. Dev. 34, 111, 1990); that they are the correctly rounded values is
// checked for every one of the 2^24 uniforms.  The paired sweep is issue-bound
// (74 % of the slots); with this, its two slots' normals together, and one clamp
// per cell, 67M particles of N = 64 went from 14.55 to 13.17 ms for 16 cycles.
__device__ __forceinline__ void radius_pair(uint32_t ra, uint32_t rb, float& rad_a, float& rad_b) {
  const uint32_t k[2] = {ra >> 8, rb >> 8};
  const unsigned long long C = f2_both(5.9604644775390625e-8f);
  const unsigned long long K = f2_pack(__uint2float_rn(k[0]), __uint2float_rn(k[1]));
  float u[2], v[2], m[2], f[2], ef[2], g[2], h[2];
  f2_unpack(f2_fma_rn(K, C, f2_both(2.98023223876953125e-8f)), u[0], u[1]);
  // v = 1 - u from 2^24 - k, exact in FP32
  const unsigned long long V = f2_fma_rn(f2_fma_rn(K, f2_both(-1.f), f2_both(16777216.f)), C,
                                         f2_both(-2.98023223876953125e-8f));
  f2_unpack(V, v[0], v[1]);
  f2_unpack(f2_fma_rn(V, f2_both(-2.f), f2_both(1.f)), h[0], h[1]);
#pragma unroll
  for (int j = 0; j < 2; ++j) {   // lower half: u = 2^e m, m in [sqrt(1/2), sqrt(2))
    const uint32_t b = __float_as_uint(u[j]);
    m[j] = __uint_as_float((b & 0x007FFFFFu) | 0x3F800000u);
    const bool halve = m[j] >= 1.41421356237309505f;
    m[j] = halve ? 0.5f * m[j] : m[j];
    ef[j] = (float)((int)(b >> 23) - (halve ? 126 : 127));
  }
  f2_unpack(f2_add_rn(f2_pack(m[0], m[1]), f2_both(-1.f)), g[0], g[1]);
#pragma unroll
  for (int j = 0; j < 2; ++j) {   // upper half: e = 0 above sqrt(1/2), else -1
    const bool upper = k[j] >= (1u << 23), e0 = v[j] <= 0.29289321881345248f;
    f[j] = upper ? (e0 ? -v[j] : h[j]) : g[j];
    ef[j] = upper ? (e0 ? 0.f : -1.f) : ef[j];
  }
  // s = f/(2 + f)
  const unsigned long long F = f2_pack(f[0], f[1]);
  const unsigned long long ND = f2_fma_rn(F, f2_both(-1.f), f2_both(-2.f));   // -(2 + f)
  float nd[2], y[2];
  f2_unpack(ND, nd[0], nd[1]);
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y[0]) : "f"(-nd[0]));
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y[1]) : "f"(-nd[1]));
  const unsigned long long Y0 = f2_pack(y[0], y[1]);
  const unsigned long long Y = f2_fma_rn(f2_fma_rn(ND, Y0, f2_both(1.f)), Y0, Y0);
  const unsigned long long Q = f2_mul_rn(F, Y);
  const unsigned long long S = f2_fma_rn(f2_fma_rn(ND, Q, F), Y, Q);
  // log1p_reduced
  const unsigned long long Z = f2_mul_rn(S, S);
  unsigned long long T = f2_fma_rn(Z, f2_both(0.111111111111111111f), f2_both(0.142857142857142857f));
  T = f2_fma_rn(Z, T, f2_both(0.2f));
  T = f2_fma_rn(Z, T, f2_both(0.333333333333333333f));
  const unsigned long long SS = f2_add_rn(S, S);
  const unsigned long long L1 = f2_fma_rn(f2_mul_rn(SS, Z), T, SS);
  const unsigned long long EF = f2_pack(ef[0], ef[1]);
  const unsigned long long L = f2_fma_rn(EF, f2_both(0.693145751953125f),
                                         f2_fma_rn(EF, f2_both(1.428606820309417232e-6f), L1));
  // sqrt(x), x = -2 ln u >= 2^-24
  const unsigned long long X = f2_mul_rn(L, f2_both(-2.f)), NX = f2_mul_rn(L, f2_both(2.f));
  float x[2], w[2];
  f2_unpack(X, x[0], x[1]);
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(w[0]) : "f"(x[0]));
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(w[1]) : "f"(x[1]));
  const unsigned long long W = f2_pack(w[0], w[1]);
  const unsigned long long G = f2_mul_rn(X, W), NG = f2_mul_rn(NX, W), H = f2_mul_rn(W, f2_both(0.5f));
  const unsigned long long E = f2_fma_rn(NG, H, f2_both(0.5f));
  const unsigned long long G1 = f2_fma_rn(G, E, G), NG1 = f2_fma_rn(NG, E, NG), H1 = f2_fma_rn(H, E, H);
  f2_unpack(f2_fma_rn(f2_fma_rn(NG1, G1, X), H1, G1), rad_a, rad_b);
}

// The three standard normals of two smart Monte Carlo moves, each from its one
// draw r: Box-Muller of the uniforms of the top 24 bits of (x, y) and (z, w),
// the radius from the accurate log (a small absolute error of ln u near u = 1
// would be a large one of the radius), the angle by the hardware sincos.
__device__ __forceinline__ void smc_normals2(const uint4& r, const uint4& t, float g[3], float h[3]) {
  float a0, b0, a1, b1, sn, cs;
  radius_pair(r.x, t.x, a0, b0);
  radius_pair(r.z, t.z, a1, b1);
  sincos_2pi_uniform_fast(r.y, &sn, &cs);
  g[0] = a0 * cs;
  g[1] = a0 * sn;
  sincos_2pi_uniform_fast(r.w, &sn, &cs);
  g[2] = a1 * cs;
  sincos_2pi_uniform_fast(t.y, &sn, &cs);
  h[0] = b0 * cs;
  h[1] = b0 * sn;
  sincos_2pi_uniform_fast(t.w, &sn, &cs);
  h[2] = b1 * cs;
}

// The same for one move.
__device__ __forceinline__ void smc_normals(const uint4& r, float& gx, float& gy, float& gz) {
  float a0, a1, sn, cs;
  radius_pair(r.x, r.z, a0, a1);
  sincos_2pi_uniform_fast(r.y, &sn, &cs);
  gx = a0 * cs;
  gy = a0 * sn;
  sincos_2pi_uniform_fast(r.w, &sn, &cs);
  gz = a1 * cs;
}

}  // namespace soma
