// Counter-based Gaussian draws on the device.
//
// Philox4x32-10 (Salmon, Moraes, Dror & Shaw, "Parallel random numbers: as
// easy as 1, 2, 3", SC'11): a 128-bit counter and a 64-bit key, ten rounds of
// two 32x32->64 multiplications (multipliers 0xD2511F53, 0xCD9E8D57) with the
// key bumped by the Weyl constants 0x9E3779B9, 0xBB67AE85 between rounds.
//
// Uniforms: (floor(w / 2^9) + 1/2) / 2^23, exact in FP32, inside (0, 1).
// Gaussians: Box-Muller, evaluated in FP32 with explicitly rounded
// operations so that every implementation of this specification returns the
// same bits:
//   ln u  : u = m 2^e, m in [sqrt(1/2), sqrt(2)); s = (m-1)/(m+1);
//           ln m = 2 s (1 + z/3 + z^2/5 + z^3/7 + z^4/9), z = s^2 (Horner,
//           fused multiply-adds, innermost first: 1/9 * z + 1/7);
//           ln u = e * (1420/2048) + (e * tail + ln m)
//   sin/cos 2 pi u: t = 4u, q = rint(t), r = t - q, th = r * (pi/2);
//           sin th, cos th by Taylor polynomials in z = th^2 to degree 9 and
//           10; the result rotated by q quarter turns.
#pragma once
#include <stdint.h>

#include "fx.cuh"

namespace pdfgb {

__device__ __forceinline__ void philox4x32_10(uint32_t c[4], uint32_t k0, uint32_t k1) {
#pragma unroll
  for (int r = 0; r < 10; ++r) {
    const uint32_t lo0 = 0xD2511F53u * c[0];
    const uint32_t hi0 = __umulhi(0xD2511F53u, c[0]);
    const uint32_t lo1 = 0xCD9E8D57u * c[2];
    const uint32_t hi1 = __umulhi(0xCD9E8D57u, c[2]);
    const uint32_t n0 = hi1 ^ c[1] ^ k0;
    const uint32_t n2 = hi0 ^ c[3] ^ k1;
    c[0] = n0;
    c[1] = lo1;
    c[2] = n2;
    c[3] = lo0;
    k0 += 0x9E3779B9u;
    k1 += 0xBB67AE85u;
  }
}

// (floor(w / 2^9) + 1/2) 2^-23: the 23 bits as the mantissa of a float in
// [2^23, 2^24), less 2^23 - 1/2 (exact).
__device__ __forceinline__ float u01_from_word(uint32_t w) {
  return __fmul_rn(__fsub_rn(__uint_as_float(0x4B000000u | (w >> 9)), 8388607.5f), 0x1p-23f);
}
__device__ __forceinline__ fx::f2 u01_from_words(uint32_t w1, uint32_t w2) {
  const fx::f2 t = {__uint_as_float(0x4B000000u | (w1 >> 9)), __uint_as_float(0x4B000000u | (w2 >> 9))};
  return fx::mul2(fx::sub2(t, fx::dup2(8388607.5f)), fx::dup2(0x1p-23f));
}

// u = m 2^e with m in [0.70710678, 1.41421356): the difference to the bits of
// 0.70710678 carries e in its exponent field.  Returns m; e as a float in the
// low bits of 12582912 + e.
__device__ __forceinline__ float split_unit(float u, float* e_magic) {
  const uint32_t bits = __float_as_uint(u);
  const int e = (int)(bits - 0x3F3504F3u) >> 23;
  *e_magic = __uint_as_float(0x4B400000u + (uint32_t)e);
  return __uint_as_float(bits - ((uint32_t)e << 23));
}

// ln u for u in [2^-24, 1): normal FP32 input only.
__device__ __forceinline__ float ln_unit(float u) {
  float em;
  const float m = split_unit(u, &em);
  const float s = __fdiv_rn(__fsub_rn(m, 1.0f), __fadd_rn(m, 1.0f));
  const float z = __fmul_rn(s, s);
  float p = __fmaf_rn(z, 1.0f / 9.0f, 1.0f / 7.0f);
  p = __fmaf_rn(p, z, 1.0f / 5.0f);
  p = __fmaf_rn(p, z, 1.0f / 3.0f);
  p = __fmaf_rn(p, z, 1.0f);
  const float lnm = __fmul_rn(__fmul_rn(2.0f, s), p);
  const float fe = __fsub_rn(em, 12582912.0f);
  return __fmaf_rn(fe, 1420.0f / 2048.0f, __fmaf_rn(fe, -2.12194440054690582e-4f, lnm));
}

// ln_unit and sincos_2pi of two values, lane by lane the same operations.
__device__ __forceinline__ fx::f2 ln_unit2(fx::f2 u) {
  using namespace fx;
  f2 em, m;
  m.x = split_unit(u.x, &em.x);
  m.y = split_unit(u.y, &em.y);
  const f2 n = sub2(m, dup2(1.0f)), d = add2(m, dup2(1.0f));
  const f2 s = {__fdiv_rn(n.x, d.x), __fdiv_rn(n.y, d.y)};
  const f2 z = mul2(s, s);
  f2 p = fma2(z, dup2(1.0f / 9.0f), dup2(1.0f / 7.0f));
  p = fma2(p, z, dup2(1.0f / 5.0f));
  p = fma2(p, z, dup2(1.0f / 3.0f));
  p = fma2(p, z, dup2(1.0f));
  const f2 lnm = mul2(mul2(dup2(2.0f), s), p);
  const f2 fe = sub2(em, dup2(12582912.0f));
  return fma2(fe, dup2(1420.0f / 2048.0f), fma2(fe, dup2(-2.12194440054690582e-4f), lnm));
}

// sin and cos of the quadrant (the low bits of 12582912 + q) from those of
// the reduced angle: exchanged in odd quadrants, signs by quadrant.
__device__ __forceinline__ void quadrant(float q_magic, float s, float c, float* sn, float* cs) {
  const uint32_t q = __float_as_uint(q_magic);
  const float a = (q & 1u) ? c : s, b = (q & 1u) ? s : c;
  *sn = __uint_as_float(__float_as_uint(a) ^ ((q << 30) & 0x80000000u));
  *cs = __uint_as_float(__float_as_uint(b) ^ (((q + 1u) << 30) & 0x80000000u));
}

__device__ __forceinline__ void sincos_2pi(float u, float* sn, float* cs) {
  const float t = __fmul_rn(4.0f, u);
  const float qm = __fadd_rn(t, 12582912.0f);  // nearest integer, ties to even
  const float r = __fsub_rn(t, __fsub_rn(qm, 12582912.0f));
  const float th = __fmul_rn(r, 1.57079632679489662f);
  const float z = __fmul_rn(th, th);
  float ps = __fmaf_rn(z, 1.0f / 362880.0f, -1.0f / 5040.0f);
  ps = __fmaf_rn(ps, z, 1.0f / 120.0f);
  ps = __fmaf_rn(ps, z, -1.0f / 6.0f);
  ps = __fmaf_rn(ps, z, 1.0f);
  const float s = __fmul_rn(th, ps);
  float pc = __fmaf_rn(z, -1.0f / 3628800.0f, 1.0f / 40320.0f);
  pc = __fmaf_rn(pc, z, -1.0f / 720.0f);
  pc = __fmaf_rn(pc, z, 1.0f / 24.0f);
  pc = __fmaf_rn(pc, z, -0.5f);
  const float c = __fmaf_rn(pc, z, 1.0f);
  quadrant(qm, s, c, sn, cs);
}

__device__ __forceinline__ void sincos_2pi2(fx::f2 u, fx::f2* sn, fx::f2* cs) {
  using namespace fx;
  const f2 t = mul2(dup2(4.0f), u);
  const f2 qm = add2(t, dup2(12582912.0f));
  const f2 r = sub2(t, sub2(qm, dup2(12582912.0f)));
  const f2 th = mul2(r, dup2(1.57079632679489662f));
  const f2 z = mul2(th, th);
  f2 ps = fma2(z, dup2(1.0f / 362880.0f), dup2(-1.0f / 5040.0f));
  ps = fma2(ps, z, dup2(1.0f / 120.0f));
  ps = fma2(ps, z, dup2(-1.0f / 6.0f));
  ps = fma2(ps, z, dup2(1.0f));
  const f2 s = mul2(th, ps);
  f2 pc = fma2(z, dup2(-1.0f / 3628800.0f), dup2(1.0f / 40320.0f));
  pc = fma2(pc, z, dup2(-1.0f / 720.0f));
  pc = fma2(pc, z, dup2(1.0f / 24.0f));
  pc = fma2(pc, z, dup2(-0.5f));
  const f2 c = fma2(pc, z, dup2(1.0f));
  quadrant(qm.x, s.x, c.x, &sn->x, &cs->x);
  quadrant(qm.y, s.y, c.y, &sn->y, &cs->y);
}

__device__ __forceinline__ void box_muller(uint32_t w1, uint32_t w2, float* g0, float* g1) {
  const float rad = __fsqrt_rn(__fmul_rn(-2.0f, ln_unit(u01_from_word(w1))));
  float sn, cs;
  sincos_2pi(u01_from_word(w2), &sn, &cs);
  *g0 = __fmul_rn(rad, cs);
  *g1 = __fmul_rn(rad, sn);
}

// Four N(0,1) from the block with counter (c0, c1, c2, c3).
__device__ __forceinline__ void gauss4(uint64_t seed, uint32_t c0, uint32_t c1, uint32_t c2,
                                       uint32_t c3, float g[4]) {
  uint32_t c[4] = {c0, c1, c2, c3};
  philox4x32_10(c, (uint32_t)seed, (uint32_t)(seed >> 32));
  // the two Box-Muller pairs lane by lane: the same bits as box_muller twice
  const fx::f2 ln = fx::mul2(fx::dup2(-2.0f), ln_unit2(u01_from_words(c[0], c[2])));
  fx::f2 sn, cs;
  sincos_2pi2(u01_from_words(c[1], c[3]), &sn, &cs);
  const fx::f2 rad = {__fsqrt_rn(ln.x), __fsqrt_rn(ln.y)};
  const fx::f2 gc = fx::mul2(rad, cs), gs = fx::mul2(rad, sn);
  g[0] = gc.x;
  g[1] = gs.x;
  g[2] = gc.y;
  g[3] = gs.y;
}

enum : uint32_t { kPurposeStep = 0, kPurposeInit = 1, kPurposeRedist = 2 };

}  // namespace pdfgb
