// Per-site arithmetic of the axisymmetric Shan-Chen LBM step (arXiv:1310.1871,
// Sec. II and App. A) on explicitly rounded lane types, shared by the step
// kernels of every schedule.  Every kernel that includes this header is compiled
// with -fmad=false and states each fused multiply-add itself, so that every
// schedule computes a site with the same operations and gets the same bits.
#pragma once

#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <stdint.h>

#include <type_traits>

#include "amlbm.h"
#include "amlbm_internal.cuh"

namespace amlbm {
namespace {

// D2Q9 velocities (c_z, c_r), weights, specular (r-flipped) and reversed directions.
__host__ __device__ constexpr int cz_(int i) {
  return (i == 1 || i == 5 || i == 8) ? 1 : (i == 3 || i == 6 || i == 7) ? -1 : 0;
}
__host__ __device__ constexpr int cr_(int i) {
  return (i == 2 || i == 5 || i == 6) ? 1 : (i == 4 || i == 7 || i == 8) ? -1 : 0;
}
__host__ __device__ constexpr double w_(int i) {
  return i == 0 ? 4.0 / 9.0 : (i < 5 ? 1.0 / 9.0 : 1.0 / 36.0);
}
__host__ __device__ constexpr int mirror_(int i) {
  return i == 2 ? 4 : i == 4 ? 2 : i == 5 ? 8 : i == 8 ? 5 : i == 6 ? 7 : i == 7 ? 6 : i;
}
__host__ __device__ constexpr int opp_(int i) {
  return i == 0 ? 0 : i == 1 ? 3 : i == 3 ? 1 : i == 2 ? 4 : i == 4 ? 2
       : i == 5 ? 7 : i == 7 ? 5 : i == 6 ? 8 : 6;
}

// ---------------------------------------------------------------- lanes --
struct F1 { float v; };
struct D1 { double v; };

__device__ __forceinline__ F1 operator+(F1 a, F1 b) { return {__fadd_rn(a.v, b.v)}; }
__device__ __forceinline__ F1 operator-(F1 a, F1 b) { return {__fsub_rn(a.v, b.v)}; }
__device__ __forceinline__ F1 operator*(F1 a, F1 b) { return {__fmul_rn(a.v, b.v)}; }
__device__ __forceinline__ F1 operator-(F1 a) { return {-a.v}; }
__device__ __forceinline__ F1 fma(F1 a, F1 b, F1 c) { return {__fmaf_rn(a.v, b.v, c.v)}; }

__device__ __forceinline__ D1 operator+(D1 a, D1 b) { return {__dadd_rn(a.v, b.v)}; }
__device__ __forceinline__ D1 operator-(D1 a, D1 b) { return {__dsub_rn(a.v, b.v)}; }
__device__ __forceinline__ D1 operator*(D1 a, D1 b) { return {__dmul_rn(a.v, b.v)}; }
__device__ __forceinline__ D1 operator-(D1 a) { return {-a.v}; }
__device__ __forceinline__ D1 fma(D1 a, D1 b, D1 c) { return {__fma_rn(a.v, b.v, c.v)}; }

// FP64 runs at 1/58 of the FP32 rate on GB300 (measured: one warp instruction per
// 16.4 clocks and SM), so an FP64 step costs what its FP64 operations cost and
// nothing else.  The FP64 form therefore evaluates the same equations with fewer
// of them: the stencils without their common factors (folded into the force and
// source constants), the equilibrium, collision and sources of opposite directions
// from one symmetric and one antisymmetric part, no arithmetic in its codec:
// 214 operations per site against 472 in the two-kernel schedule.  The FP32
// forms keep their own sequence of operations.
template <class T> constexpr bool kWide = std::is_same<T, D1>::value;

template <class T> struct Lane;
template <> struct Lane<F1> { using C = float; static constexpr int N = 1; };
template <> struct Lane<D1> { using C = double; static constexpr int N = 1; };

template <class T> __device__ __forceinline__ T lit(double c);
template <> __device__ __forceinline__ F1 lit<F1>(double c) { return {float(c)}; }
template <> __device__ __forceinline__ D1 lit<D1>(double c) { return {c}; }

// Reciprocal and exponential.  FP32 uses the correctly rounded
// reciprocal and the SFU exponential (relative error ~1e-7, far below the
// storage rounding); FP64 the correctly rounded reciprocal and exp.
__device__ __forceinline__ F1 rcp(F1 a) { return {__frcp_rn(a.v)}; }
__device__ __forceinline__ D1 rcp(D1 a) { return {__drcp_rn(a.v)}; }
__device__ __forceinline__ F1 expl(F1 a) { return {__expf(a.v)}; }
__device__ __forceinline__ D1 expl(D1 a) { return {exp(a.v)}; }

// ------------------------------------------------------------- storage --
// Storage codecs: conversion between the stored element and the arithmetic
// type.  The shift W_i s of the FP32 / 16-bit forms is applied by the callers
// (decode: f = q + W_i s; encode: q = f - W_i s).  IEEE half holds q * 2^10 so
// that the shifted populations (down to ~1e-7) stay in its normal range; the
// power-of-two scale is exact.  from_sr rounds stochastically with the random
// word x: its top bits are added to the bits below the stored precision and the
// sum is truncated, so a value rounds up with probability equal to its distance
// from the lower neighbour (unbiased in expectation).
template <class S> struct Store;
template <> struct Store<double> {
  using C = double;
  using T = D1;
  static __device__ __forceinline__ C to(double v) { return v; }
  static __device__ __forceinline__ double from(C v) { return v; }
  static __device__ __forceinline__ double from_sr(C v, uint32_t) { return v; }
};
template <> struct Store<float> {
  using C = float;
  using T = F1;
  static __device__ __forceinline__ C to(float v) { return v; }
  static __device__ __forceinline__ float from(C v) { return v; }
  static __device__ __forceinline__ float from_sr(C v, uint32_t) { return v; }
};
template <> struct Store<__half> {
  using C = float;
  using T = F1;
  static __device__ __forceinline__ C to(__half v) { return __half2float(v) * (1.0f / 1024.0f); }
  static __device__ __forceinline__ __half from(C v) { return __float2half_rn(v * 1024.0f); }
  static __device__ __forceinline__ __half from_sr(C v, uint32_t x) {
    // FP32 keeps 13 more mantissa bits than FP16 (for FP16-normal values)
    const uint32_t b = __float_as_uint(v * 1024.0f) + (x >> 19);
    return __float2half_rz(__uint_as_float(b));
  }
};
template <> struct Store<__nv_bfloat16> {
  using C = float;
  using T = F1;
  static __device__ __forceinline__ C to(__nv_bfloat16 v) { return __bfloat162float(v); }
  static __device__ __forceinline__ __nv_bfloat16 from(C v) { return __float2bfloat16_rn(v); }
  static __device__ __forceinline__ __nv_bfloat16 from_sr(C v, uint32_t x) {
    // bfloat16 is the upper half of the FP32 bit pattern
    const uint32_t b = __float_as_uint(v) + (x >> 16);
    return __ushort_as_bfloat16((unsigned short)(b >> 16));
  }
};

__device__ __forceinline__ float fma_c(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ double fma_c(double a, double b, double c) { return __fma_rn(a, b, c); }

// Random words of the stochastic rounding.  Each site seeds its own stream with
// an integer hash of (site, step): the xorshift-multiply mixer with shifts
// 16, 15, 16 and multipliers 0x7feb352d, 0x846ca68b published by C. Wellons
// ("lowbias32", hash-prospector, 2018); the nine
// populations then take successive states of the linear congruential generator
// x <- 1664525 x + 1013904223 (mod 2^32) (Knuth / Numerical Recipes constants),
// whose top bits are the ones the codecs use.
__device__ __forceinline__ uint32_t mix32(uint32_t x) {
  x ^= x >> 16;
  x *= 0x7feb352dU;
  x ^= x >> 15;
  x *= 0x846ca68bU;
  x ^= x >> 16;
  return x;
}
__device__ __forceinline__ uint32_t lcg_next(uint32_t x) { return x * 1664525u + 1013904223u; }

// Shift s of a site from its stored psi: 0 (none), rho_ref (global), or the
// density recovered from psi, -rho0 ln(1 - psi/rho0) (local).  Writer and
// reader evaluate it from the same stored psi with the same non-contracted
// operations, so both see the same s bit for bit.
__device__ __forceinline__ double shift_base(int mode, double psi, double inv_rho0, double rho0,
                                             double rref) {
  (void)psi; (void)inv_rho0; (void)rho0;
  return mode == 1 ? rref : 0.0;  // FP64 storage is never shifted locally
}
__device__ __forceinline__ float shift_base(int mode, float psi, float inv_rho0, float rho0,
                                            float rref) {
  if (mode >= 2) {
    const float q = __fsub_rn(1.0f, __fmul_rn(psi, inv_rho0));
    return __fmul_rn(-rho0, __logf(q));
  }
  return mode == 1 ? rref : 0.0f;
}

__device__ __forceinline__ int wrapz(int k, int Nz) {
  k %= Nz;
  return k < 0 ? k + Nz : k;
}
// Row whose value a ghost row mirrors (about r = 0 and r = Nr), clamped so that
// rows deeper than any stencil reaches still address real memory.
__device__ __forceinline__ int reflect_row(int j, int Nr) {
  if (j < 0) j = -1 - j;
  if (j >= Nr) j = 2 * Nr - 1 - j;
  return j < 0 ? 0 : (j >= Nr ? Nr - 1 : j);
}
// The same with inlet and outlet rows, whose ghosts mirror about the boundary
// row itself (zero normal derivative of psi there).
__device__ __forceinline__ int ghost_row(int j, int Nr, bool inlet, bool outlet) {
  if (j < 0) j = inlet ? -j : -1 - j;
  if (j >= Nr) j = outlet ? 2 * (Nr - 1) - j : 2 * Nr - 1 - j;
  return j < 0 ? 0 : (j >= Nr ? Nr - 1 : j);
}
// Column of a ghost column: periodic wrap, or the mirror about the walls at
// z = -1/2 and z = Nz - 1/2 (clamped like the rows).
__device__ __forceinline__ int ghost_col(int k, int Nz, bool walls) {
  if (!walls) return wrapz(k, Nz);
  if (k < 0) k = -1 - k;
  if (k >= Nz) k = 2 * Nz - 1 - k;
  return k < 0 ? 0 : (k >= Nz ? Nz - 1 : k);
}

// ------------------------------------------------------------- physics --
// Isotropic 4th-order first derivative along r, Sec. II.D Eq. forthorder_firstderivativex:
//   d_r phi(x) = (1/36) sum_i c_ir (8 phi(x + c_i) - phi(x + 2 c_i)).
// p points at x in a row-major tile whose rows (r) are `st` apart.  The terms
// are added in z-mirror pairs (c_5, c_6), (c_8, c_7) so that a field mirrored
// in z gives an exactly mirrored derivative: without this, the rounding of the
// FP32 forms carries a net axial bias every step and a drop drifts along the
// axis.
template <class T>
__device__ __forceinline__ T link8(const T* p, int dz, int dr, int st) {
  return fma(lit<T>(8.0), p[dr * st + dz], -p[2 * dr * st + 2 * dz]);
}
// The FP64 form returns 36 times the derivative.
template <class T>
__device__ __forceinline__ T iso_r(const T* p, int st) {
  const T a = link8(p, 0, 1, st) - link8(p, 0, -1, st);
  const T b = (link8(p, 1, 1, st) + link8(p, -1, 1, st)) - (link8(p, 1, -1, st) + link8(p, -1, -1, st));
  if constexpr (kWide<T>) return a + b;
  else return (a + b) * lit<T>(1.0 / 36.0);
}
// 1D 4th-order central difference with element step `step` (Sec. II.D): the
// inner and outer operators of d_zr psi, and the velocity gradients of the
// sources.  (The velocity gradients do not take the isotropic stencil: its
// diagonal taps reverse the sign of d_r u_z on a mode alternating in z, and
// mu d_r u_z / r then amplifies that mode next to a no-slip wall.)
// The FP64 form returns 12 times the difference.
template <class T>
__device__ __forceinline__ T d1(const T* p, int step) {
  const T d = fma(lit<T>(8.0), p[step] - p[-step], -(p[2 * step] - p[-2 * step]));
  if constexpr (kWide<T>) return d;
  else return d * lit<T>(1.0 / 12.0);
}
// The derivatives themselves from what iso_r, d1, sc_sums and their compositions
// return (for the adjoint's stored intermediates).
template <class T>
__device__ __forceinline__ T unscale(T v, double factor) {
  if constexpr (kWide<T>) return v * lit<T>(1.0 / factor);
  else return v;
}

// c_i . v of direction i
template <class T>
__device__ __forceinline__ T cdot(int i, T vz, T vr) {
  switch (i) {
    case 1: return vz;
    case 2: return vr;
    case 3: return -vz;
    case 4: return -vr;
    case 5: return vz + vr;
    case 6: return vr - vz;
    case 7: return -(vz + vr);
    default: return vz - vr;
  }
}
// rho = sum_i f_i and j = sum_i c_i f_i, added in z-mirror pairs.
template <class T>
__device__ __forceinline__ T moment0(const T* f) {
  return (f[0] + (f[2] + f[4])) + ((f[1] + f[3]) + ((f[5] + f[6]) + (f[7] + f[8])));
}
template <class T>
__device__ __forceinline__ T moment_z(const T* f) {
  return (f[1] - f[3]) + ((f[5] - f[6]) + (f[8] - f[7]));
}
template <class T>
__device__ __forceinline__ T moment_r(const T* f) {
  return (f[2] - f[4]) + ((f[5] - f[8]) + (f[6] - f[7]));
}
// The nine equilibria (Eq. feq; W_i rho (1 + 3 c.v + 4.5 (c.v)^2 - 1.5 v^2))
// with f^eq_0 = rho - sum_{i>0} f^eq_i: the same value in exact arithmetic, but
// the collision then conserves mass to rounding.  With the directly evaluated
// f^eq_0 the FP32-rounded weights do not sum to 1 and the FP32 forms gain mass
// every step (a 1.5e-5 drift over 1000 steps of the static drop, and a 1e-4
// density error at the interface).
template <class T>
__device__ __forceinline__ void equilibrium(T rho, T vz, T vr, T* fe) {
  const T A = fma(fma(vz, vz, vr * vr), lit<T>(-1.5), lit<T>(1.0));
  const T r9 = rho * lit<T>(1.0 / 9.0), r36 = rho * lit<T>(1.0 / 36.0);
#pragma unroll
  for (int i = 1; i < 9; ++i) {
    const T cv = cdot(i, vz, vr);
    fe[i] = (i < 5 ? r9 : r36) * fma(fma(cv, lit<T>(4.5), lit<T>(3.0)), cv, A);
  }
  fe[0] = rho - ((fe[2] + fe[4]) + ((fe[1] + fe[3]) + ((fe[5] + fe[6]) + (fe[7] + fe[8]))));
}
// h_i = W_i (S + (c_iz H_z + c_ir H_r) / c_s^2), Eq. condition_h, with
// h_0 = S - sum_{i>0} h_i, so that sum_i h_i = S to rounding (the App. A
// zeroth moment) in every precision.
template <class T>
__device__ __forceinline__ void sources(T S_, T Hz, T Hr, T* h) {
  const T z3 = Hz * lit<T>(3.0), r3 = Hr * lit<T>(3.0);
#pragma unroll
  for (int i = 1; i < 9; ++i) h[i] = lit<T>(w_(i)) * (S_ + cdot(i, z3, r3));
  h[0] = S_ - ((h[2] + h[4]) + ((h[1] + h[3]) + ((h[5] + h[6]) + (h[7] + h[8]))));
}
// Discrete force of the Guo forcing (Guo, Zheng & Shi 2002):
//   s_i = W_i (3 (c_i . F - u . F) + 9 (c_i . u)(c_i . F)),
// with s_0 = -sum_{i>0} s_i (zeroth moment 0 to rounding; first moment F).
template <class T>
__device__ __forceinline__ void guo_force(T uz, T ur, T Fz, T Fr, T* s) {
  const T uF = fma(uz, Fz, ur * Fr);
#pragma unroll
  for (int i = 1; i < 9; ++i) {
    const T cF = cdot(i, Fz, Fr), cu = cdot(i, uz, ur);
    s[i] = lit<T>(w_(i)) * fma(cu * lit<T>(9.0), cF, (cF - uF) * lit<T>(3.0));
  }
  s[0] = -((s[2] + s[4]) + ((s[1] + s[3]) + ((s[5] + s[6]) + (s[7] + s[8]))));
}
// Shan-Chen neighbour sums sum_i W_i psi(x + c_i) c_i (Eq. scforce) around p; the
// FP64 form returns 36 times them, from the differences along the two diagonals.
template <class T>
__device__ __forceinline__ void sc_sums(const T* p, int Z, T& sz, T& sr) {
  if constexpr (kWide<T>) {
    const T u = p[Z + 1] - p[-Z - 1], w = p[-Z + 1] - p[Z - 1];
    sz = fma(p[1] - p[-1], lit<T>(4.0), u + w);
    sr = fma(p[Z] - p[-Z], lit<T>(4.0), u - w);
    return;
  }
  sz = fma(p[1] - p[-1], lit<T>(1.0 / 9.0),
           ((p[Z + 1] - p[Z - 1]) + (p[-Z + 1] - p[-Z - 1])) * lit<T>(1.0 / 36.0));
  sr = fma(p[Z] - p[-Z], lit<T>(1.0 / 9.0),
           ((p[Z + 1] - p[-Z + 1]) + (p[Z - 1] - p[-Z - 1])) * lit<T>(1.0 / 36.0));
}
// The instance constants of the step in the lane type.
template <class T>
struct Par {
  T tau, omega, negG, gfac, gz, rho0, inv_rho0, cmu;
};
// The FP64 form's constants: -G / 36, -G / (18 * 1296), 1 - 1/tau, 1/(9 tau),
// (tau - 1/2) / 36 and -rho0, next to the ones both use.
template <>
struct Par<D1> {
  D1 tau, gz, inv_rho0, rho0, negG36, gf1296, om1, om9, cmu12;
};
__device__ __forceinline__ float kc(const InstDesc& D, int c, float) { return D.k32[c]; }
__device__ __forceinline__ double kc(const InstDesc& D, int c, double) { return D.k64[c]; }
template <class T>
__device__ __forceinline__ T splat(typename Lane<T>::C c);
template <> __device__ __forceinline__ F1 splat<F1>(float c) { return {c}; }
template <> __device__ __forceinline__ D1 splat<D1>(double c) { return {c}; }
// q.gfac = -(G / 2) c_s^4 with c_s^4 = 1/9; q.cmu = mu / rho = c_s^2 (tau - 1/2)
template <class T>
__device__ __forceinline__ Par<T> par_of(const InstDesc& D) {
  using C = typename Lane<T>::C;
  Par<T> q;
  q.tau = splat<T>(kc(D, K_TAU, C()));
  if constexpr (kWide<T>) {
    q.gz = splat<T>(D.k64[K_GZ]);
    q.inv_rho0 = splat<T>(D.k64[K_INVRHO0]);
    q.rho0 = splat<T>(D.k64[K_RHO0]);
    q.negG36 = splat<T>(D.k64[K_NEGG36]);
    q.gf1296 = splat<T>(D.k64[K_GF1296]);
    q.om1 = splat<T>(D.k64[K_OM1]);
    q.om9 = splat<T>(D.k64[K_OM9]);
    q.cmu12 = splat<T>(D.k64[K_CMU12]);
    return q;
  } else {
  q.omega = splat<T>(kc(D, K_OMEGA, C()));
  q.negG = splat<T>(kc(D, K_NEGG, C()));
  q.gfac = splat<T>(kc(D, K_GFAC, C()));
  q.gz = splat<T>(kc(D, K_GZ, C()));
  q.rho0 = splat<T>(kc(D, K_RHO0, C()));
  q.inv_rho0 = splat<T>(kc(D, K_INVRHO0, C()));
  q.cmu = splat<T>(kc(D, K_CMU, C()));
  return q;
  }
}
// 1 / r of row j, r = j + r0 with r0 = r_off + 1/2 the radius of row 0 (the sum
// is exact in either precision for the half-integer radii of the workloads)
__device__ __forceinline__ F1 inv_r_of(F1, int j, float r0) { return rcp(F1{__int2float_rn(j) + r0}); }
__device__ __forceinline__ D1 inv_r_of(D1, int j, double r0) { return rcp(D1{__int2double_rn(j) + r0}); }

// What the site arithmetic needs of row j besides its index: 1 / r and, in the FP64
// form, the force factors that carry the stencils' scales (formed once per row or
// per site with the same operations).
template <class T>
struct Row {
  T inv_r;
};
template <>
struct Row<D1> {
  D1 g, g9, inv36;    // of the force: -G/(18 1296) / r, 9 times that, 36 / r
  D1 inv12, i3, ni9;  // of the sources: 12 / r, 1 / (3 r), -1 / (9 r)
};
template <class T>
__device__ __forceinline__ Row<T> row_of(const Par<T>& q, int j, typename Lane<T>::C r0) {
  Row<T> w;
  const T inv_r = inv_r_of(T(), j, r0);
  if constexpr (kWide<T>) {
    w.g = q.gf1296 * inv_r;
    w.g9 = w.g * lit<T>(9.0);
    w.inv36 = inv_r * lit<T>(36.0);
    w.inv12 = inv_r * lit<T>(12.0);
    w.i3 = inv_r * lit<T>(1.0 / 3.0);
    w.ni9 = inv_r * lit<T>(-1.0 / 9.0);
  } else {
    w.inv_r = inv_r;
  }
  return w;
}

// The force of Eq. scforce and Eq. scAxisExtra without the body force rho g_z,
// from sc_sums, iso_r (dr0), iso_r of that (Drr) and d1 along z of d1 along r (Dzr).
template <class T>
__device__ __forceinline__ void forces_partial(const Par<T>& q, T psi, T sz, T sr, bool ax, T dr0, T Drr, T Dzr,
                                               const Row<T>& w, T& Fz, T& Fr) {
  if constexpr (kWide<T>) {
    const T gpsi = psi * q.negG36;
    Fz = gpsi * sz;
    Fr = gpsi * sr;
    if (ax) {
      Fz = fma(psi * w.g9, Dzr, Fz);
      Fr = fma(psi * w.g, fma(-dr0, w.inv36, Drr), Fr);
    }
  } else {
    const T gpsi = psi * q.negG;
    Fz = gpsi * sz;
    Fr = gpsi * sr;
    if (ax) {
      const T g = (psi * q.gfac) * w.inv_r;
      Fz = fma(g, Dzr, Fz);
      Fr = fma(g, fma(-dr0, w.inv_r, Drr), Fr);
    }
  }
}
// Total force on a site (Eq. scforce, Eq. scAxisExtra, body force rho g_z).
template <class T>
__device__ __forceinline__ void forces(const Par<T>& q, T rho, T psi, T sz, T sr, bool ax, T dr0, T Drr,
                                       T Dzr, const Row<T>& w, T& Fz, T& Fr) {
  forces_partial(q, psi, sz, sr, ax, dr0, Drr, Dzr, w, Fz, Fr);
  Fz = fma(rho, q.gz, Fz);
}

// The BGK collision of a site (Eq. lbm2d): f + (f^eq - f)/tau at u^eq = v, with the
// Guo forcing f^eq at u plus gk = 1 - 1/(2 tau) times the discrete force.  put(i, value)
// receives the nine populations.
//
// FP64: with m = rho / (9 tau), the populations of a pair of opposite directions are
// (1 - 1/tau) f + q +- k, q = W/(1/9) m (1 - 1.5 v^2 + 4.5 (c.v)^2) and k the part odd
// in c; the Guo force adds to both parts.  The rest population takes what the others leave
// of rho (rest_of), so that a collision keeps the site's mass to the rounding of one sum:
// evaluated directly, with factors (1 - 1/tau) and 1/(9 tau) whose shares do not sum to one
// in 53 bits and an m rounded the same way every step where the state is steady, a
// 64 x 32 drop loses 2.4e-12 of its mass in 40,000 steps (closed: 1.2e-15), and the
// gradients of the drop's shape carry up to 50 times the error.
template <class T>
__device__ __forceinline__ T rest_of(T rho, T pair_z, T pair_r, T pair_s, T pair_d) {
  return rho - (pair_r + (pair_z + (pair_s + pair_d)));
}
template <class T, class PUT>
__device__ __forceinline__ void collide(const Par<T>& q, bool guo, T gk, const T* f, T rho, T uz, T ur, T jz, T jr,
                                        T Fz, T Fr, T inv_rho, PUT&& put) {
  if constexpr (kWide<T>) {
    T vz = uz, vr = ur;
    if (!guo) {
      vz = fma(Fz, q.tau, jz) * inv_rho;
      vr = fma(Fr, q.tau, jr) * inv_rho;
    }
    const T m9 = rho * q.om9;
    T a9 = m9 * fma(fma(vz, vz, vr * vr), lit<T>(-1.5), lit<T>(1.0));
    const T c9 = m9 * lit<T>(4.5), k3 = m9 * lit<T>(3.0);
    T kz = k3 * vz, kr = k3 * vr;
    const T sv = vz + vr, dv = vr - vz;
    T ez = c9 * vz, er = c9 * vr, es = c9 * sv, ed = c9 * dv;
    if (guo) {
      const T g3 = gk * lit<T>(1.0 / 3.0);
      a9 = fma(-g3, fma(uz, Fz, ur * Fr), a9);
      kz = fma(g3, Fz, kz);
      kr = fma(g3, Fr, kr);
      ez = fma(gk, Fz, ez);
      er = fma(gk, Fr, er);
      es = fma(gk, Fz + Fr, es);
      ed = fma(gk, Fr - Fz, ed);
    }
    const T quarter = lit<T>(0.25);
    const T qz = fma(ez, vz, a9), qr = fma(er, vr, a9);
    const T qs = fma(es, sv, a9), qd = fma(ed, dv, a9), ks = kz + kr, kd = kr - kz;
    // each pair is put as it is formed: only the sums stay live
    auto pair = [&](int a, T up, int b, T down) {
      const T ga = fma(q.om1, f[a], up), gb = fma(q.om1, f[b], down);
      put(a, ga);
      put(b, gb);
      return ga + gb;
    };
    const T pz = pair(1, qz + kz, 3, qz - kz);
    const T pr = pair(2, qr + kr, 4, qr - kr);
    const T ps = pair(5, (qs + ks) * quarter, 7, (qs - ks) * quarter);
    const T pd = pair(6, (qd + kd) * quarter, 8, (qd - kd) * quarter);
    put(0, rest_of(rho, pz, pr, ps, pd));
  } else {
    T fe[9];
    if (guo) {
      equilibrium(rho, uz, ur, fe);
      T sg[9];
      guo_force(uz, ur, Fz, Fr, sg);
#pragma unroll
      for (int i = 0; i < 9; ++i) put(i, fma(sg[i], gk, fma(fe[i] - f[i], q.omega, f[i])));
    } else {
      const T vz = fma(Fz, q.tau, jz) * inv_rho, vr = fma(Fr, q.tau, jr) * inv_rho;
      equilibrium(rho, vz, vr, fe);
#pragma unroll
      for (int i = 0; i < 9; ++i) put(i, fma(fe[i] - f[i], q.omega, f[i]));
    }
  }
}

// Axisymmetric sources of App. A at a site: S = -rho u_r / r,
// H_z = (mu (d_r u_z + d_z u_r) - rho u_r u_z) / r,
// H_r = (2 mu (d_r u_r - u_r / r) - rho u_r^2) / r.
// The FP64 form returns S / 9, H_z / 3 and H_r / 3, the terms of h_i of the axis
// directions, from 12 times the gradients.
template <class T>
__device__ __forceinline__ void site_sources(const Par<T>& q, T rho, T uz, T ur, T druz, T dzur, T drur,
                                             const Row<T>& w, T& S_, T& Hz, T& Hr) {
  if constexpr (kWide<T>) {
    const T mu = rho * q.cmu12, rur = rho * ur;
    S_ = rur * w.ni9;
    Hz = fma(mu, druz + dzur, -(rur * uz)) * w.i3;
    Hr = fma(mu * lit<T>(2.0), fma(-ur, w.inv12, drur), -(rur * ur)) * w.i3;
  } else {
    const T mu = rho * q.cmu, rur = rho * ur;
    S_ = -(rur * w.inv_r);
    Hz = fma(mu, druz + dzur, -(rur * uz)) * w.inv_r;
    Hr = fma(mu * lit<T>(2.0), fma(-ur, w.inv_r, drur), -(rur * ur)) * w.inv_r;
  }
}
// f + h_i of one direction in the FP64 form, from what site_sources returns
// (h_i = W_i (S + 3 c_i . H), Eq. condition_h).
__device__ __forceinline__ D1 add_source(int i, D1 f, D1 S9, D1 Z, D1 R) {
  const D1 quarter = lit<D1>(0.25);
  switch (i) {
    case 0: return fma(lit<D1>(4.0), S9, f);
    case 1: return f + (S9 + Z);
    case 2: return f + (S9 + R);
    case 3: return f + (S9 - Z);
    case 4: return f + (S9 - R);
    case 5: return fma(quarter, S9 + (Z + R), f);
    case 6: return fma(quarter, S9 + (R - Z), f);
    case 7: return fma(quarter, S9 - (Z + R), f);
    default: return fma(quarter, S9 - (R - Z), f);
  }
}
// psi = rho0 (1 - exp(-rho / rho0)), Eq. psi.
template <class T>
__device__ __forceinline__ T psi_of(const Par<T>& q, T rho) {
  if constexpr (kWide<T>) return fma(-q.rho0, expl(-rho * q.inv_rho0), q.rho0);
  return (lit<T>(1.0) - expl(-rho * q.inv_rho0)) * q.rho0;
}

// Decode the nine populations of a site from their stored values q[i]:
// f_i = q_i + W_i s (shift modes 0-2, one fused multiply-add) or, in the
// equilibrium mode (3), f_i = q_i + f^eq_i(s, v) with the stored velocity
// v = (vz, vr).
template <class S, class T>
__device__ __forceinline__ void decode_values(int mode, const S* q, typename Store<S>::C psi,
                                              typename Store<S>::C vz, typename Store<S>::C vr,
                                              typename Store<S>::C inv_rho0, typename Store<S>::C rho0,
                                              typename Store<S>::C rref, T* f) {
  if constexpr (kWide<T>) {  // FP64 storage holds f itself
#pragma unroll
    for (int i = 0; i < 9; ++i) f[i] = T{q[i]};
    return;
  }
  const T sbt{shift_base(mode, psi, inv_rho0, rho0, rref)};
  if (mode == 3) {
    T fe[9];
    equilibrium(sbt, T{vz}, T{vr}, fe);
#pragma unroll
    for (int i = 0; i < 9; ++i) f[i] = T{Store<S>::to(q[i])} + fe[i];
  } else {
#pragma unroll
    for (int i = 0; i < 9; ++i) f[i] = fma(lit<T>(w_(i)), sbt, T{Store<S>::to(q[i])});
  }
}

// The same from global memory: q[i * plane], and in the equilibrium mode the
// velocity in the two planes that follow psi (pv points at the site's psi).
template <class S, class T>
__device__ __forceinline__ void decode_site(int mode, const S* q, size_t plane, typename Store<S>::C psi,
                                            const typename Store<S>::C* pv, typename Store<S>::C inv_rho0,
                                            typename Store<S>::C rho0, typename Store<S>::C rref, T* f) {
  using C = typename Store<S>::C;
  S qv[9];
#pragma unroll
  for (int i = 0; i < 9; ++i) qv[i] = q[i * plane];
  const C vz = mode == 3 ? pv[plane] : C(0), vr = mode == 3 ? pv[2 * plane] : C(0);
  decode_values<S>(mode, qv, psi, vz, vr, inv_rho0, rho0, rref, f);
}

// The stored values of the new populations fn of a site: q_i = fn_i - W_i s
// (shift modes 0-2) or, in the equilibrium mode, q_i = fn_i - f^eq_i(s, v) with
// the bare velocity v = sum_i c_i fn_i / rho of the new state (returned in
// vz, vr); 16-bit stores round to nearest or (rounding != 0) stochastically
// with words drawn from (site, step).
template <class S, class T>
__device__ __forceinline__ void encode_values(int mode, const T* fn, T rho, typename Store<S>::C psi,
                                              typename Store<S>::C inv_rho0, typename Store<S>::C rho0,
                                              typename Store<S>::C rref, int rounding, uint32_t site,
                                              uint32_t step, S* q, typename Store<S>::C& vz_out,
                                              typename Store<S>::C& vr_out) {
  using C = typename Store<S>::C;
  if constexpr (kWide<T>) {
#pragma unroll
    for (int i = 0; i < 9; ++i) q[i] = fn[i].v;
    vz_out = vr_out = C(0);
    return;
  }
  const C sb = shift_base(mode, psi, inv_rho0, rho0, rref);
  C fv[9], base[9];
#pragma unroll
  for (int i = 0; i < 9; ++i) fv[i] = fn[i].v;
  if (mode == 3) {
    const T ir = rcp(rho), vz = moment_z(fn) * ir, vr = moment_r(fn) * ir;
    T fe[9];
    equilibrium(T{sb}, vz, vr, fe);
#pragma unroll
    for (int i = 0; i < 9; ++i) base[i] = fv[i] - fe[i].v;
    vz_out = vz.v;
    vr_out = vr.v;
  } else {
#pragma unroll
    for (int i = 0; i < 9; ++i) base[i] = fma_c(C(-w_(i)), sb, fv[i]);
    vz_out = C(0);
    vr_out = C(0);
  }
  if (sizeof(S) == 2 && rounding) {
    uint32_t x = mix32(site ^ mix32(step + 0x9E3779B9u));
#pragma unroll
    for (int i = 0; i < 9; ++i) {
      x = lcg_next(x);
      q[i] = Store<S>::from_sr(base[i], x);
    }
  } else {
#pragma unroll
    for (int i = 0; i < 9; ++i) q[i] = Store<S>::from(base[i]);
  }
}

// Store the new populations fn of a site and its psi (at *pso); in the
// equilibrium mode also the bare velocity v of the new state (after psi).
template <class S, class T>
__device__ __forceinline__ void encode_site(int mode, S* o, typename Store<S>::C* pso, size_t plane,
                                            const T* fn, T rho, typename Store<S>::C psi,
                                            typename Store<S>::C inv_rho0, typename Store<S>::C rho0,
                                            typename Store<S>::C rref, int rounding, uint32_t site,
                                            uint32_t step) {
  using C = typename Store<S>::C;
  S q[9];
  C vz, vr;
  encode_values<S>(mode, fn, rho, psi, inv_rho0, rho0, rref, rounding, site, step, q, vz, vr);
#pragma unroll
  for (int i = 0; i < 9; ++i) o[i * plane] = q[i];
  if (mode == 3) {
    pso[plane] = vz;
    pso[2 * plane] = vr;
  }
  pso[0] = psi;
}

}  // namespace
}  // namespace amlbm
