// Packed FP32 lanes for the strip kernel: F2 holds the values of two adjacent z-sites
// and operates on both with one instruction (add, sub, mul and fma .f32x2 of sm_100
// and later).  Each lane rounds as the scalar operation does, so a function evaluated
// on F2 gives the bits of the same function on F1.  On GB300 a packed operation takes
// the FP32 pipe as long as its two scalar ones (measured: 1.90 packed against 3.55
// scalar warp instructions per clock and SM) but one issue slot.  (What then bounds the
// strips stands in amlbm_step_strip.cu.)
//
// A packed operand has no negation, so the specialisations below state the functions
// of amlbm_physics.cuh with their negations moved into constants, differences and
// signs of products; negation is exact, so the results are the same bits (up to the
// sign of a zero).
#pragma once

#include "amlbm_physics.cuh"

namespace amlbm {
namespace {

struct F2 { unsigned long long v; };

template <> struct Lane<F2> { using C = float; static constexpr int N = 2; };

__device__ __forceinline__ F2 pack(float a, float b) {
  F2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ void unpack(F2 x, float& a, float& b) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(x.v));
}
__device__ __forceinline__ float lo(F2 x) { float a, b; unpack(x, a, b); return a; }
__device__ __forceinline__ float hi(F2 x) { float a, b; unpack(x, a, b); return b; }

__device__ __forceinline__ F2 operator+(F2 a, F2 b) {
  F2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
  return r;
}
__device__ __forceinline__ F2 operator-(F2 a, F2 b) {
  F2 r;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
  return r;
}
__device__ __forceinline__ F2 fma(F2 a, F2 b, F2 c) {
  F2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(c.v));
  return r;
}
// The product as a fused multiply-add to zero (the same value up to the sign of a zero):
// a mul.rn.f32x2 that feeds an add.rn.f32x2 is contracted by the assembler of CUDA 13.0
// into one rounding, which the scalar operations never are.
__device__ __forceinline__ F2 operator*(F2 a, F2 b) {
  F2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(0ull));
  return r;
}
template <> __device__ __forceinline__ F2 lit<F2>(double c) {
  const unsigned b = __float_as_uint(float(c));
  return {((unsigned long long)b << 32) | b};
}
template <> __device__ __forceinline__ F2 splat<F2>(float c) { return pack(c, c); }
__device__ __forceinline__ F2 negate(F2 x) {  // only where no constant can take the sign
  F2 r;
  asm("xor.b64 %0, %1, 0x8000000080000000;" : "=l"(r.v) : "l"(x.v));
  return r;
}

// Correctly rounded reciprocal: an approximate one, one Newton step, and the correction
// step that rounds correctly (P. Markstein, "Computation of elementary functions on the
// IBM RISC System/6000 processor", 1990) where neither argument nor result leaves
// the normal range; __frcp_rn, whose value it equals (tested for every argument),
// elsewhere.  __frcp_rn everywhere costs about 14 issue slots and 78 clocks each.
__device__ __forceinline__ bool rcp_plain(float x) {  // 2^-125 <= |x| < 2^125
  return ((__float_as_uint(x) & 0x7fffffffu) - 0x01000000u) < 0x7d000000u;
}
__device__ __forceinline__ float rcp_start(float x) {
  float y;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float rcp_one(float x) {
  if (!rcp_plain(x)) return __frcp_rn(x);
  float y = rcp_start(x);
  y = __fmaf_rn(__fmaf_rn(-x, y, 1.0f), y, y);
  return __fmaf_rn(__fmaf_rn(-x, y, 1.0f), y, y);
}
__device__ __forceinline__ F2 rcp(F2 x) {
  float a, b;
  unpack(x, a, b);
  if (rcp_plain(a) && rcp_plain(b)) {
    const F2 nx = x * lit<F2>(-1.0), one = lit<F2>(1.0);
    F2 y = pack(rcp_start(a), rcp_start(b));
    y = fma(fma(nx, y, one), y, y);
    return fma(fma(nx, y, one), y, y);
  }
  return pack(__frcp_rn(a), __frcp_rn(b));
}

// The instance constants with the signs the packed functions need.
template <>
struct Par<F2> {
  F2 tau, omega, negG, gfac, gz, rho0, neg_inv_rho0, neg_cmu;
};
template <>
__device__ __forceinline__ Par<F2> par_of<F2>(const InstDesc& D) {
  Par<F2> q;
  q.tau = splat<F2>(D.k32[K_TAU]);
  q.omega = splat<F2>(D.k32[K_OMEGA]);
  q.negG = splat<F2>(D.k32[K_NEGG]);
  q.gfac = splat<F2>(D.k32[K_GFAC]);
  q.gz = splat<F2>(D.k32[K_GZ]);
  q.rho0 = splat<F2>(D.k32[K_RHO0]);
  q.neg_inv_rho0 = splat<F2>(-D.k32[K_INVRHO0]);
  q.neg_cmu = splat<F2>(-D.k32[K_CMU]);
  return q;
}

// psi = rho0 (1 - exp(-rho / rho0))
template <>
__device__ __forceinline__ F2 psi_of<F2>(const Par<F2>& q, F2 rho) {
  float a, b;
  unpack(rho * q.neg_inv_rho0, a, b);
  return (lit<F2>(1.0) - pack(__expf(a), __expf(b))) * q.rho0;
}

// equilibrium(): for c . v = -w the two negations of (4.5 c.v + 3) c.v + A are taken
// by -(4.5 w - 3) w = (4.5 w - 3)(-w).
template <>
__device__ __forceinline__ void equilibrium<F2>(F2 rho, F2 vz, F2 vr, F2* fe) {
  const F2 A = fma(fma(vz, vz, vr * vr), lit<F2>(-1.5), lit<F2>(1.0));
  const F2 r9 = rho * lit<F2>(1.0 / 9.0), r36 = rho * lit<F2>(1.0 / 36.0);
  const F2 c45 = lit<F2>(4.5), p3 = lit<F2>(3.0), m3 = lit<F2>(-3.0);
  const F2 s = vz + vr, d = vr - vz;  // c_5 . v = -c_7 . v and c_6 . v = -c_8 . v
  fe[1] = r9 * fma(fma(vz, c45, p3), vz, A);
  fe[3] = r9 * fma(fma(vz, c45, m3), vz, A);
  fe[2] = r9 * fma(fma(vr, c45, p3), vr, A);
  fe[4] = r9 * fma(fma(vr, c45, m3), vr, A);
  fe[5] = r36 * fma(fma(s, c45, p3), s, A);
  fe[7] = r36 * fma(fma(s, c45, m3), s, A);
  fe[6] = r36 * fma(fma(d, c45, p3), d, A);
  fe[8] = r36 * fma(fma(d, c45, m3), d, A);
  fe[0] = rho - ((fe[2] + fe[4]) + ((fe[1] + fe[3]) + ((fe[5] + fe[6]) + (fe[7] + fe[8]))));
}

// f + h_i of all nine directions (sources(), site_sources()): nir = -1/r.
__device__ __forceinline__ void add_sources(const Par<F2>& q, F2 rho, F2 uz, F2 ur, F2 druz, F2 dzur, F2 drur,
                                            F2 nir, F2* f) {
  const F2 nmu = rho * q.neg_cmu, rur = rho * ur;
  const F2 S = rur * nir;
  const F2 Hz = fma(nmu, druz + dzur, rur * uz) * nir;
  const F2 Hr = fma(nmu * lit<F2>(2.0), fma(ur, nir, drur), rur * ur) * nir;
  const F2 z3 = Hz * lit<F2>(3.0), r3 = Hr * lit<F2>(3.0);
  const F2 s = z3 + r3, d = r3 - z3, w9 = lit<F2>(w_(1)), w36 = lit<F2>(w_(5));
  F2 h[9];
  h[1] = w9 * (S + z3);
  h[2] = w9 * (S + r3);
  h[3] = w9 * (S - z3);
  h[4] = w9 * (S - r3);
  h[5] = w36 * (S + s);
  h[6] = w36 * (S + d);
  h[7] = w36 * (S - s);
  h[8] = w36 * (S - d);
  h[0] = S - ((h[2] + h[4]) + ((h[1] + h[3]) + ((h[5] + h[6]) + (h[7] + h[8]))));
#pragma unroll
  for (int i = 0; i < 9; ++i) f[i] = f[i] + h[i];
}

// guo_force() without its negations: cF - uF for c . F = -w is -(w + uF).
template <>
__device__ __forceinline__ void guo_force<F2>(F2 uz, F2 ur, F2 Fz, F2 Fr, F2* s) {
  const F2 uF = fma(uz, Fz, ur * Fr), nine = lit<F2>(9.0), three = lit<F2>(3.0), m3 = lit<F2>(-3.0);
  const F2 us = uz + ur, ud = ur - uz, Fs = Fz + Fr, Fd = Fr - Fz;
  auto up = [&](double w, F2 u, F2 F) { return lit<F2>(w) * fma(u * nine, F, (F - uF) * three); };
  auto down = [&](double w, F2 u, F2 F) { return lit<F2>(w) * fma(u * nine, F, (F + uF) * m3); };
  s[1] = up(w_(1), uz, Fz);
  s[2] = up(w_(2), ur, Fr);
  s[3] = down(w_(3), uz, Fz);
  s[4] = down(w_(4), ur, Fr);
  s[5] = up(w_(5), us, Fs);
  s[6] = up(w_(6), ud, Fd);
  s[7] = down(w_(7), us, Fs);
  s[8] = down(w_(8), ud, Fd);
  s[0] = lit<F2>(0.0) - ((s[2] + s[4]) + ((s[1] + s[3]) + ((s[5] + s[6]) + (s[7] + s[8]))));
}

}  // namespace
}  // namespace amlbm
