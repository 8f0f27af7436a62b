// Counter-based normal generator shared by the proxy samplers: Philox4x64-10
// (Salmon, Moraes, Dror, Shaw, SC'11) and the Box-Muller transform (Box and
// Muller 1958) in float32.
#pragma once

#include <stdint.h>

#include "umma.cuh"

namespace mmshift {
namespace {

// Philox4x64-10 (Salmon et al., SC'11): multipliers and Weyl key increments.
constexpr uint64_t kPhM0 = 0xD2E7470EE14C6C93ull;
constexpr uint64_t kPhM1 = 0xCA5A826395121157ull;
constexpr uint64_t kPhW0 = 0x9E3779B97F4A7C15ull;
constexpr uint64_t kPhW1 = 0xBB67AE8584CAA73Bull;

__device__ __forceinline__ void philox4x64_10(uint64_t c[4], uint64_t k0, uint64_t k1) {
#pragma unroll
  for (int rnd = 0; rnd < 10; ++rnd) {
    if (rnd) { k0 += kPhW0; k1 += kPhW1; }
    const uint64_t hi0 = __umul64hi(kPhM0, c[0]), lo0 = kPhM0 * c[0];
    const uint64_t hi1 = __umul64hi(kPhM1, c[2]), lo1 = kPhM1 * c[2];
    const uint64_t n0 = hi1 ^ c[1] ^ k0, n2 = hi0 ^ c[3] ^ k1;
    c[0] = n0; c[1] = lo1; c[2] = n2; c[3] = lo0;
  }
}

// Uniform in (0, 1) from a 32-bit word: ((w >> 9) + 1/2) 2^-23, exact in float.
__device__ __forceinline__ float uniform_of(uint32_t w) {
  return ((float)(w >> 9) + 0.5f) * 1.1920928955078125e-07f;
}

// Pairs of float32 in packed operations, each half rounded like the scalar
// operation, so two uniforms' transforms share their instructions (the samplers
// are bound by issue). With two instead of four draws unrolled, proxy stage of
// the 28-layer 32K stack, N = 512: 240 -> 212 us, of the 8K stack with a 64-query
// window 252 -> 233 us. (A hand-written 64 x 64-bit product of four 32-bit ones
// was slower than the compiler's, 252 -> 269 us.)
using F2 = uint64_t;
__device__ __forceinline__ F2 f2(float x) { return umma::pk2(x, x); }
__device__ __forceinline__ F2 mul2(F2 a, F2 b) {
  F2 d;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}

// ln(u) for two uniforms u in (0, 1): u = m 2^e with m in [sqrt(1/2), sqrt(2)),
// ln m = 2 atanh(s) with s = (m - 1) / (m + 1) (|s| <= 0.1716; m - 1 is exact,
// 1 / (m + 1) from the approximate reciprocal and one Newton step, about one
// ulp) from the series 2 (s + s^3/3 + ... + s^13/13), whose truncation is
// below 2e-12 relative, and e ln 2 with ln 2 split into a short leading part
// (its product with e is exact) and the remainder (the argument reduction of
// Cody and Waite, 1980). Rounding leaves about 3 float32 ulp of relative
// error.
__device__ __forceinline__ void split_uniform(float u, float& m, float& e, float& rcp) {
  const uint32_t bits = __float_as_uint(u);
  int ei = (int)(bits >> 23) - 127;
  m = __uint_as_float((bits & 0x7FFFFFu) | 0x3F800000u);   // [1, 2)
  if (m > 1.41421356f) { m *= 0.5f; ++ei; }
  e = (float)ei;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(rcp) : "f"(m + 1.0f));
}
__device__ __forceinline__ F2 ln_uniform2(float u0, float u1) {
  float m0, m1, e0, e1, r0, r1;
  split_uniform(u0, m0, e0, r0);
  split_uniform(u1, m1, e1, r1);
  const F2 m = umma::pk2(m0, m1), fe = umma::pk2(e0, e1);
  F2 rcp = umma::pk2(r0, r1);
  const F2 nden = umma::pk2(-(m0 + 1.0f), -(m1 + 1.0f));
  rcp = umma::ffma2(rcp, umma::ffma2(nden, rcp, f2(1.0f)), rcp);
  const F2 s = mul2(umma::fadd2(m, f2(-1.0f)), rcp);
  const F2 t = mul2(s, s);
  F2 p = f2(1.0f / 13.0f);
  p = umma::ffma2(p, t, f2(1.0f / 11.0f));
  p = umma::ffma2(p, t, f2(1.0f / 9.0f));
  p = umma::ffma2(p, t, f2(1.0f / 7.0f));
  p = umma::ffma2(p, t, f2(1.0f / 5.0f));
  p = umma::ffma2(p, t, f2(1.0f / 3.0f));
  const F2 s2 = mul2(f2(2.0f), s);
  const F2 lnm = umma::ffma2(mul2(s2, t), p, s2);
  return umma::ffma2(fe, f2(0.693145751953125f), umma::ffma2(fe, f2(1.4286068203094172e-06f), lnm));
}

// sin(pi x), cos(pi x) for two |x| < 1, x a multiple of 2^-23: x = y + k/2
// with k = rint(2x) and |y| <= 1/4 (both exact), Taylor polynomials of
// sin t and cos t at t = pi y (|t| <= pi/4; truncation below 1e-11), then
// the quarter-turn rotation by k.
__device__ __forceinline__ void quarter_turns(float k, float s0, float c0, float& sn, float& cs) {
  const int q = ((int)k) & 3;                     // quarter turns
  const float sa = (q & 1) ? c0 : s0, ca = (q & 1) ? s0 : c0;
  sn = (q & 2) ? -sa : sa;
  cs = (q == 1 || q == 2) ? -ca : ca;
}
__device__ __forceinline__ void sincos_pi2(float x0, float x1, float (&sn)[2], float (&cs)[2]) {
  const float k0 = rintf(2.0f * x0), k1 = rintf(2.0f * x1);
  const F2 y = umma::ffma2(f2(-0.5f), umma::pk2(k0, k1), umma::pk2(x0, x1));
  const F2 t = mul2(y, f2(3.14159265358979323846f));
  const F2 t2 = mul2(t, t);
  F2 ps = f2(-1.0f / 39916800.0f);                            // -1/11!
  ps = umma::ffma2(ps, t2, f2(1.0f / 362880.0f));             //  1/9!
  ps = umma::ffma2(ps, t2, f2(-1.0f / 5040.0f));              // -1/7!
  ps = umma::ffma2(ps, t2, f2(1.0f / 120.0f));                //  1/5!
  ps = umma::ffma2(ps, t2, f2(-1.0f / 6.0f));                 // -1/3!
  const F2 s0 = umma::ffma2(mul2(ps, t2), t, t);
  F2 pc = f2(1.0f / 479001600.0f);                            //  1/12!
  pc = umma::ffma2(pc, t2, f2(-1.0f / 3628800.0f));           // -1/10!
  pc = umma::ffma2(pc, t2, f2(1.0f / 40320.0f));              //  1/8!
  pc = umma::ffma2(pc, t2, f2(-1.0f / 720.0f));               // -1/6!
  pc = umma::ffma2(pc, t2, f2(1.0f / 24.0f));                 //  1/4!
  pc = umma::ffma2(pc, t2, f2(-0.5f));                        // -1/2!
  const F2 c0 = umma::ffma2(pc, t2, f2(1.0f));
  float sa, sb, ca, cb;
  umma::upk2(s0, sa, sb);
  umma::upk2(c0, ca, cb);
  quarter_turns(k0, sa, ca, sn[0], cs[0]);
  quarter_turns(k1, sb, cb, sn[1], cs[1]);
}

// Box-Muller on two pairs: sqrt(-2 ln u) (cos 2 pi v, sin 2 pi v) in float32
// from the low and high halves of two 64-bit words, with 2v reduced to (-1, 1)
// exactly before the rotation.
__device__ __forceinline__ float reduced_turns(uint32_t c) {
  const float v2 = 2.0f * uniform_of(c);              // 2v in (0, 2), exact
  return v2 >= 1.0f ? v2 - 2.0f : v2;                 // exact
}
__device__ __forceinline__ void box_muller2(uint64_t a, uint64_t b, float* z) {
  float l0, l1, sn[2], cs[2];
  umma::upk2(mul2(f2(-2.0f), ln_uniform2(uniform_of((uint32_t)a), uniform_of((uint32_t)b))), l0, l1);
  sincos_pi2(reduced_turns((uint32_t)(a >> 32)), reduced_turns((uint32_t)(b >> 32)), sn, cs);
  const float r0 = sqrtf(l0), r1 = sqrtf(l1);
  z[0] = r0 * cs[0];
  z[1] = r0 * sn[0];
  z[2] = r1 * cs[1];
  z[3] = r1 * sn[1];
}

// Eight standard normals from one Philox4x64-10 draw with counter
// (c0, c1, b, layer) and key (k0, k1): its 64-bit outputs split low word first
// into eight uniforms, Box-Muller on consecutive pairs. The query-space
// sampler uses c0 = i * d/8 + q, c1 = query head, key (seed, 0); the
// hidden-space sampler c0 = i * d_model/8 + q, c1 = 0, key (seed, 1).
__device__ __forceinline__ void normals8_at(uint64_t c0, uint64_t c1, int b, int layer,
                                            uint64_t k0, uint64_t k1, float (&z)[8]) {
  uint64_t c[4] = {c0, c1, (uint64_t)b, (uint64_t)(int64_t)layer};
  philox4x64_10(c, k0, k1);
  box_muller2(c[0], c[1], z);
  box_muller2(c[2], c[3], z + 4);
}

}  // namespace
}  // namespace mmshift
