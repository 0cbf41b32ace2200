// Discrete adjoint of the axisymmetric Shan-Chen LBM step (the reverse sweep of
// the update of Sec. II, transposed operation by operation), the device map from
// Legendre shape amplitudes to the initial drop, the objectives, and the
// checkpointed driver behind amlbm_adjoint / amlbm_objective.
//
// The forward intermediates of every state of a checkpoint segment are written
// while the segment is recomputed (launch_step_inter: the step and the
// intermediates of the state it starts from).  One adjoint step (lambda^{n+1} ->
// lambda^n, state f^n) then runs as two kernels:
//   adj_local : mu = transpose of the streaming map (a gather); the adjoints of the
//               sources' velocity gradients on the tile and two sites around it; then
//               per site the adjoint of the BGK collision and of the sources S, H_z,
//               H_r, the transposed gradient stencils, the adjoint of
//               u = (j + F/2)/rho and u^eq = (j + tau F)/rho, of F_SC (Eq. scforce) and
//               F^gamma (Eq. scAxisExtra); G and tau parts
//   adj_psi   : transposed 1D d_z (of d_zr) and isotropic d_r (of d_rr) on the tile and
//               two sites around it; then the transposed Shan-Chen neighbour sum, 1D d_r
//               and isotropic d_r on psi, d psi/d rho, and
//               lambda^n_i = (1 - omega) mu_i + rho_bar + c_i . j_bar
// (four kernels and 30 planes of intermediates before: the small lattices of these
// runs are bound by the chain of launches and memory round trips, FP64 by its
// operations).  Ghost rows: a field mirrored with sign s about a boundary and read by
// a stencil that is antisymmetric (symmetric) in r has as transpose the stencil's own
// transpose on the adjoint field mirrored with sign -s (s), so the folds of the ghost rows
// need no terms of their own.  All kernels are gathers (no atomics): the sweep is
// deterministic.
//
// Collision: with the moments M0 = sum W mu, M = sum W c mu, MM = sum W c c mu of the
// gathered mu (less its value at rest, which takes the cancellation out of the tau part), the
// adjoint of f^eq is a quadratic form in u^eq: 65 operations instead of nine separate terms
// (about 190).
//
// Measured (GB300, ncu, one backward step, cold caches; the four kernels before): FP32,
// 512 x 128: 21 us (45); FP64, 256 x 128: 36 us (68), 279 FP64 operations per site (543).
// A gradient of the differentiable drop, 512 x 128, T = 100, checkpoints every 10, FP32:
// 2.5 ms (5.2; 2.8 with the forward steps on the persistent tiles); 256 x 128, T = 50, FP64: 3.9 ms (5.6).

#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <string>
#include <vector>

#include "amlbm.h"
#include "amlbm_internal.cuh"
#include "amlbm_launch.cuh"

namespace amlbm {
namespace {

__host__ __device__ constexpr int acz(int i) {
  return (i == 1 || i == 5 || i == 8) ? 1 : (i == 3 || i == 6 || i == 7) ? -1 : 0;
}
__host__ __device__ constexpr int acr(int i) {
  return (i == 2 || i == 5 || i == 6) ? 1 : (i == 4 || i == 7 || i == 8) ? -1 : 0;
}
__host__ __device__ constexpr double aw(int i) {
  return i == 0 ? 4.0 / 9.0 : (i < 5 ? 1.0 / 9.0 : 1.0 / 36.0);
}
__host__ __device__ constexpr int amirror(int i) {
  return i == 2 ? 4 : i == 4 ? 2 : i == 5 ? 8 : i == 8 ? 5 : i == 6 ? 7 : i == 7 ? 6 : i;
}
__host__ __device__ constexpr int aopp(int i) {
  return i == 0 ? 0 : i == 1 ? 3 : i == 3 ? 1 : i == 2 ? 4 : i == 4 ? 2
       : i == 5 ? 7 : i == 7 ? 5 : i == 6 ? 8 : 6;
}

// Periodic wrap of a column that lies a few sites outside [0, Nz) (no
// division: stencil offsets are at most 4 beyond a tile, so one or two corrections
// suffice unless Nz is smaller than that).
__device__ __forceinline__ int wz(int k, int Nz) {
  while (k < 0) k += Nz;
  while (k >= Nz) k -= Nz;
  return k;
}
// The lattice row that a row up to Nr ghosts beyond the axis or the wall mirrors.
__device__ __forceinline__ int mirror_row(int j, int Nr) { return j < 0 ? -1 - j : j >= Nr ? 2 * Nr - 1 - j : j; }

template <class C>
struct Adj {
  int Nz, Nr, P, wall, axisym;
  size_t plane;
  C tau, omega, G, gz, inv_rho0;
  const C* lam_in;
  C* lam_out;
  const C* f;      // state f^n, 9 planes
  const C* inter;  // I_COUNT planes
  C *rhob, *jzb, *jrb, *psib, *qz, *qr, *dzrb, *drrb, *drdb;  // adjoints, [Nr][P] each
  double *accG, *accT;
};

template <class C>
__device__ __forceinline__ C feq_std(int i, C rho, C vz, C vr) {
  const C cv = C(acz(i)) * vz + C(acr(i)) * vr;
  return C(aw(i)) * rho * (C(1) + C(3) * cv + C(4.5) * cv * cv - C(1.5) * (vz * vz + vr * vr));
}

// mu_q at the lattice site (k, j): lambda where population q leaving it arrives
// (Sec. II.E maps).
template <class C>
__device__ __forceinline__ C arrived(const Adj<C>& A, int q, int k, int j) {
  int yk = k, yj = j + acr(q), d = q;
  if (yj < 0) {
    yj = 0; d = amirror(q);
  } else if (yj >= A.Nr) {
    yj = A.Nr - 1;
    d = A.wall == AMLBM_WALL_NOSLIP ? aopp(q) : amirror(q);
  }
  if (acz(q) != 0 && !(d == aopp(q) && yj == j)) {
    yk += acz(q);
    yk = yk < 0 ? A.Nz - 1 : yk == A.Nz ? 0 : yk;
  }
  return A.lam_in[d * A.plane + (size_t)yj * A.P + yk];
}
// 9 sum W c_z mu and 9 sum W c_r mu from mu of the eight moving populations.
template <class C>
__device__ __forceinline__ C first_z(const C* mu) {
  return (mu[1] - mu[3]) + C(0.25) * ((mu[5] - mu[7]) + (mu[8] - mu[6]));
}
template <class C>
__device__ __forceinline__ C first_r(const C* mu) {
  return (mu[2] - mu[4]) + C(0.25) * ((mu[5] - mu[7]) + (mu[6] - mu[8]));
}
// Transposes of the stencils at p, rows st apart (isotropic d_r: 36 times it; 1D
// difference with element step e: 12 times it).
template <class C>
__device__ __forceinline__ C iso_t(const C* p, int st) {
  C s = C(0);
#pragma unroll
  for (int dz = -1; dz <= 1; ++dz)
    s += C(8) * (p[-st + dz] - p[st + dz]) - (p[2 * (-st + dz)] - p[2 * (st + dz)]);
  return s;
}
template <class C>
__device__ __forceinline__ C d1_t(const C* p, int e) {
  return C(8) * (p[-e] - p[e]) - (p[-2 * e] - p[2 * e]);
}

// Tiles of ATZ x BR sites, one thread per site.
constexpr int ATZ = 32;
template <int NT, int ROWS, int W, class F>
__device__ __forceinline__ void for_region(F&& body) {
  for (int t = threadIdx.x; t < ROWS * W; t += NT) {
    const int lr = t / W;
    body(lr, t - lr * W);
  }
}

template <class C, int BR>
__global__ void __launch_bounds__(ATZ * BR) adj_local(Adj<C> A) {
  constexpr int NT = ATZ * BR, W = ATZ + 4;
  __shared__ C g1[(BR + 4) * W];    // adjoint of d_r u_z (and of d_z u_r): the tile + 2, but the corners
  __shared__ C g3[(BR + 4) * ATZ];  // adjoint of d_r u_r: rows + 2
  __shared__ C s_ir[BR + 4];        // 1 / r of rows j0 - 2 ..
  const int k0 = blockIdx.x * ATZ, j0 = blockIdx.y * BR;
  const int tx = (int)threadIdx.x % ATZ, ty = (int)threadIdx.x / ATZ, k = k0 + tx, j = j0 + ty;
  const bool in = k < A.Nz && j < A.Nr;
  const C cmu = (A.tau - C(0.5)) * C(1.0 / 3.0);
  const size_t o = (size_t)(in ? j : 0) * A.P + (in ? k : 0);
  if (threadIdx.x < BR + 4) s_ir[threadIdx.x] = C(1) / (C(mirror_row(j0 - 2 + (int)threadIdx.x, A.Nr)) + C(0.5));
  __syncthreads();
  pdl_wait();
  C mu[9];
  if (in) {
#pragma unroll
    for (int q = 0; q < 9; ++q) mu[q] = arrived(A, q, k, j);
  }
  if (A.axisym) {
    const C wall_z = A.wall == AMLBM_WALL_NOSLIP ? C(1) : C(-1);  // minus the sign u_z is mirrored with
    // g_1 = g_2 = Hz_bar mu / r, g_3 = 2 Hr_bar mu / r with H_bar = 3 sum W c mu_q
    for_region<NT, BR + 4, ATZ>([&](int lr, int lc) {
      const int y = j0 - 2 + lr, x = k0 + lc;
      if (y > A.Nr + 1 || x >= A.Nz) return;
      const int m = mirror_row(y, A.Nr);
      C v[9];
#pragma unroll
      for (int q = 1; q < 9; ++q) v[q] = arrived(A, q, x, m);
      const C c = A.inter[I_RHO * A.plane + (size_t)m * A.P + x] * (cmu * s_ir[lr]) * C(1.0 / 3.0);
      const C sz = y < 0 ? C(-1) : y >= A.Nr ? wall_z : C(1);
      g1[lr * W + lc + 2] = sz * c * first_z(v);
      g3[lr * ATZ + lc] = C(2) * c * first_r(v);
    });
    for_region<NT, BR, 4>([&](int lr, int lc) {  // two columns on either side
      const int y = j0 + lr;
      if (y >= A.Nr) return;
      const int c0 = lc < 2 ? lc : ATZ + lc, x = wz(k0 - 2 + c0, A.Nz);
      C v[9];
#pragma unroll
      for (int q = 1; q < 9; ++q)
        if (acz(q) != 0) v[q] = arrived(A, q, x, y);
      g1[(lr + 2) * W + c0] = A.inter[I_RHO * A.plane + (size_t)y * A.P + x] * (cmu * s_ir[lr + 2]) * C(1.0 / 3.0) *
                              first_z(v);
    });
    // a ragged tile: its last columns' right-hand neighbours wrap inside the tile
    if (k0 + ATZ > A.Nz) {
      for_region<NT, BR, 2>([&](int lr, int lc) {
        const int y = j0 + lr, c0 = A.Nz - k0 + lc;
        if (y >= A.Nr || c0 >= ATZ + 2) return;
        const int x = wz(A.Nz + lc, A.Nz);
        C v[9];
#pragma unroll
        for (int q = 1; q < 9; ++q)
          if (acz(q) != 0) v[q] = arrived(A, q, x, y);
        g1[(lr + 2) * W + c0 + 2] = A.inter[I_RHO * A.plane + (size_t)y * A.P + x] * (cmu * s_ir[lr + 2]) *
                                    C(1.0 / 3.0) * first_z(v);
      });
    }
    __syncthreads();
  }
  if (!in) return;
  const C* I = A.inter + o;
  const C rho = I[I_RHO * A.plane], vz = I[I_VZ * A.plane], vr = I[I_VR * A.plane];
  const C uz = I[I_UZ * A.plane], ur = I[I_UR * A.plane];
  // moments of mu - mu_0, 9 times: M0, M_z, M_r, M_zz, M_zr, M_rr.  mu is nearly the same for
  // all directions, and what is formed below depends on a constant mu only through
  // sum mu f^eq = mu_0 rho: taken of mu itself, the tau part is a difference of two sums that
  // agree to almost every bit, and term by term it keeps the rounding of f and of the weights
  // times mu.  Against an 80-bit complex-step derivative of 85 random gradients (16 x 32 to
  // 40 x 88, 8 to 50 steps), geometric mean of the relative error of dJ/dtau, term by term /
  // from mu / from mu - mu_0: FP64 1.4e-13 / 1.2e-13 / 5.7e-15, FP32 3.2e-5 / 2.4e-5 / 3.5e-6.
  // The FP32 form stays term by term in its tau part all the same: the better sums move its
  // dJ/dtau by up to 1e-3 of itself, and its results are to stay what they were.
  const C Mz = first_z(mu), Mr = first_r(mu), mu0 = mu[0];
  C dm[9];
#pragma unroll
  for (int q = 1; q < 9; ++q) dm[q] = mu[q] - mu0;
  const C pz = dm[1] + dm[3], pr = dm[2] + dm[4], ps = dm[5] + dm[7], pd = dm[6] + dm[8];
  const C diag = C(0.25) * (ps + pd);
  const C Mzz = pz + diag, Mrr = pr + diag, Mzr = C(0.25) * (ps - pd);
  const C M0 = (pz + pr) + diag;
  const C tz = vz * Mzz + vr * Mzr, tr = vz * Mzr + vr * Mrr;
  const C Aq = C(1) - C(1.5) * (vz * vz + vr * vr);
  // sum (mu - mu_0) f^eq / rho, and the adjoints of u^eq
  const C fe = C(1.0 / 9.0) * (Aq * M0 + C(4.5) * (vz * tz + vr * tr) + C(3) * (vz * Mz + vr * Mr));
  // tau part, -omega^2 sum mu (f^eq - f), of mu - mu_0 in FP64: f^eq and f both sum to rho
  C tb = C(0);
  if constexpr (sizeof(C) == 8) {
#pragma unroll
    for (int q = 1; q < 9; ++q) tb += dm[q] * A.f[q * A.plane + o];
    tb -= rho * fe;
  } else {
#pragma unroll
    for (int q = 0; q < 9; ++q) tb += mu[q] * (A.f[q * A.plane + o] - feq_std(q, rho, vz, vr));
  }
  tb *= A.omega * A.omega;
  C rb = A.omega * (mu0 + fe);
  const C com = A.omega * rho * C(1.0 / 3.0);
  const C vzb = com * (Mz + C(3) * tz - vz * M0), vrb = com * (Mr + C(3) * tr - vr * M0);
  C uzb = C(0), urb = C(0);
  const C irr = A.axisym ? s_ir[ty + 2] : C(0);
  if (A.axisym) {
    const C Sb = mu0 + C(1.0 / 9.0) * M0, Hzb = C(1.0 / 3.0) * Mz, Hrb = C(1.0 / 3.0) * Mr;
    const C d1r = I[I_G1 * A.plane] + I[I_G2 * A.plane], d3 = I[I_G3 * A.plane];
    const C muv = rho * cmu;
    // S = -rho u_r / r, H_z = (mu (g1 + g2) - rho u_r u_z) / r,
    // H_r = (2 mu (g3 - u_r / r) - rho u_r^2) / r, mu = rho (tau - 1/2) / 3
    const C hz = Hzb * irr, hr = Hrb * irr, sb = Sb * irr;
    const C e3 = d3 - ur * irr;
    const C mvb = hz * d1r + C(2) * hr * e3;
    rb += mvb * cmu - ur * (sb + hz * uz + hr * ur);
    urb = -rho * (sb + hz * uz + C(2) * hr * ur) - C(2) * hr * muv * irr;
    uzb = -rho * hz * ur;
    tb += mvb * rho * C(1.0 / 3.0);
    // transposed gradient stencils
    const C* a = g1 + (ty + 2) * W + tx + 2;
    uzb += d1_t(a, W) * C(1.0 / 12.0);
    urb += (d1_t(a, 1) + d1_t(g3 + (ty + 2) * ATZ + tx, ATZ)) * C(1.0 / 12.0);
  }
  // u = (j + F/2)/rho and u^eq = (j + tau F)/rho
  const C ir = C(1) / rho;
  const C Fz = I[I_FZ * A.plane], Fr = I[I_FR * A.plane];
  A.jzb[o] = (uzb + vzb) * ir;
  A.jrb[o] = (urb + vrb) * ir;
  const C Fzb = (C(0.5) * uzb + A.tau * vzb) * ir, Frb = (C(0.5) * urb + A.tau * vrb) * ir;
  A.rhob[o] = rb - (uzb * uz + urb * ur + vzb * vz + vrb * vr) * ir + Fzb * A.gz;
  // F_SC = -G psi s
  const C psi = I[I_PSI * A.plane];
  const C sf = Fzb * I[I_SZ * A.plane] + Frb * I[I_SR * A.plane];
  C pb = -A.G * sf;
  double gb = double(-psi * sf);
  A.qz[o] = -A.G * psi * Fzb;
  A.qr[o] = -A.G * psi * Frb;
  if (A.axisym) {
    const C gf = -A.G * C(1.0 / 18.0), gi = gf * psi * irr;
    const C t = irr * (Fzb * I[I_DZR * A.plane] + Frb * (I[I_DRR * A.plane] - I[I_DR * A.plane] * irr));
    pb += gf * t;
    gb += double(-psi * t * C(1.0 / 18.0));
    A.dzrb[o] = gi * Fzb;
    A.drrb[o] = gi * Frb;
    A.drdb[o] = -gi * Frb * irr;
  }
  A.psib[o] = pb;
  A.accG[o] += gb;
  A.accT[o] += double(tb) + double((vzb * Fz + vrb * Fr) * ir);
  pdl_trigger();
}

template <class C, int BR>
__global__ void __launch_bounds__(ATZ * BR) adj_psi(Adj<C> A) {
  constexpr int NT = ATZ * BR;
  constexpr int RZ = ATZ + 8, RR = BR + 8;  // adjoint of d_rr psi, even in r
  constexpr int DZ = ATZ + 4, DR = BR + 4;  // adjoint of d_r psi, odd in r
  constexpr int QZ = ATZ + 2, QR = BR + 2;  // adjoints of the Shan-Chen sums: z even, r odd
  __shared__ C srr[RR * RZ], szr[DR * DZ], sdr[DR * DZ], seb[DR * ATZ], sqz[QR * QZ], sqr[QR * QZ];
  __shared__ int s_col[RZ], s_off[RR];  // columns and row offsets of the tile + 4 (-1: beyond the ghost rows)
  const int k0 = blockIdx.x * ATZ, j0 = blockIdx.y * BR;
  const int tx = (int)threadIdx.x % ATZ, ty = (int)threadIdx.x / ATZ, k = k0 + tx, j = j0 + ty;
  const bool in = k < A.Nz && j < A.Nr, ax = A.axisym != 0;
  const size_t o = (size_t)(in ? j : 0) * A.P + (in ? k : 0);
  for (int i = threadIdx.x; i < RZ; i += NT) s_col[i] = wz(k0 - 4 + i, A.Nz);
  if (threadIdx.x < RR) {
    const int m = mirror_row(j0 - 4 + (int)threadIdx.x, A.Nr);
    s_off[threadIdx.x] = m < 0 || m >= A.Nr ? -1 : m * A.P;
  }
  __syncthreads();
  pdl_wait();
  C mu[9];
  if (in) {
#pragma unroll
    for (int q = 0; q < 9; ++q) mu[q] = arrived(A, q, k, j);
  }
  for_region<NT, QR, QZ>([&](int lr, int lc) {
    const int off = s_off[lr + 3], row = j0 - 1 + lr;
    if (off < 0) return;
    const int p = off + s_col[lc + 3];
    const C r = A.qr[p];
    sqz[lr * QZ + lc] = A.qz[p];
    sqr[lr * QZ + lc] = row < 0 || row >= A.Nr ? -r : r;
  });
  if (ax) {
    for_region<NT, RR, RZ>([&](int lr, int lc) {
      const int off = s_off[lr];
      if (off >= 0) srr[lr * RZ + lc] = A.drrb[off + s_col[lc]];
    });
    for_region<NT, DR, DZ>([&](int lr, int lc) {
      const int off = s_off[lr + 2];
      if (off < 0) return;
      const int p = off + s_col[lc + 2];
      szr[lr * DZ + lc] = A.dzrb[p];
      sdr[lr * DZ + lc] = A.drdb[p];
    });
    __syncthreads();
    for_region<NT, DR, DZ>([&](int lr, int lc) {
      const int row = j0 - 2 + lr;
      const bool ghost = row < 0 || row >= A.Nr;
      // a mirrored row's transpose has the mirrored sign of the row's own
      const C d = iso_t(srr + (lr + 2) * RZ + lc + 2, RZ) * C(1.0 / 36.0);
      const C own = sdr[lr * DZ + lc];
      sdr[lr * DZ + lc] = ghost ? d - own : d + own;
      if (lc >= 2 && lc < ATZ + 2) {
        const C e = d1_t(szr + lr * DZ + lc, 1) * C(1.0 / 12.0);
        seb[lr * ATZ + lc - 2] = ghost ? -e : e;
      }
    });
  }
  __syncthreads();
  if (in) {
    const C* z = sqz + (ty + 1) * QZ + tx + 1;
    const C* r = sqr + (ty + 1) * QZ + tx + 1;
    C pb = A.psib[o] +
           C(1.0 / 9.0) * ((z[-1] - z[1]) + (r[-QZ] - r[QZ])) +
           C(1.0 / 36.0) * (((z[-QZ - 1] - z[QZ + 1]) + (z[QZ - 1] - z[-QZ + 1])) +
                            ((r[-QZ - 1] - r[QZ + 1]) + (r[-QZ + 1] - r[QZ - 1])));
    if (ax) {
      pb += d1_t(seb + (ty + 2) * ATZ + tx, ATZ) * C(1.0 / 12.0);
      pb += iso_t(sdr + (ty + 2) * DZ + tx + 2, DZ) * C(1.0 / 36.0);
    }
    // d psi / d rho = exp(-rho / rho0); in FP64 1 - psi / rho0 (an exp is 20 FP64 operations),
    // whose error is 2^-53 of psi / rho0 however small the derivative is: a rounding of rho_bar
    // itself, to which it is added (gradients at rho up to 32 rho0 have the same error with
    // either)
    C dpsi;
    if constexpr (sizeof(C) == 8) dpsi = C(1) - A.inter[I_PSI * A.plane + o] * A.inv_rho0;
    else dpsi = exp(-A.inter[I_RHO * A.plane + o] * A.inv_rho0);
    const C rb = A.rhob[o] + pb * dpsi;
    const C jzb = A.jzb[o], jrb = A.jrb[o];
#pragma unroll
    for (int q = 0; q < 9; ++q)
      A.lam_out[q * A.plane + o] = (C(1) - A.omega) * mu[q] + (rb + C(acz(q)) * jzb + C(acr(q)) * jrb);
  }
  pdl_trigger();
}

// ---- the differentiable initial drop and its adjoint
// The Legendre polynomials of all amplitudes come from one upward recurrence,
// P_{m+1} = ((2m + 1) x P_m - m P_{m-1}) / (m + 1), the division as a product with a
// reciprocal from the host (one recurrence per amplitude and an FP64 division per degree
// took 295 us for the drop and 602 us for its adjoint on 512 x 128 with 16 amplitudes).
constexpr int kMaxDegree = 64;
struct DropMap {
  int Nz, Nr, l0, namp;
  double zc, R, w, rho_l, rho_v;
  double amp[32];
  double inv[kMaxDegree];  // 1 / m
};

// P_m(x) and P_{m+1}(x), advanced by one degree from m.
__device__ __forceinline__ void legendre_next(const DropMap& M, int m, double x, double& p, double& next) {
  const double q = ((2 * m + 3) * x * next - (m + 1) * p) * (m + 2 < kMaxDegree ? M.inv[m + 2] : 1.0 / (m + 2));
  p = next;
  next = q;
}
__device__ __forceinline__ void legendre_start(const DropMap& M, double x, double& p, double& next) {
  p = 1.0;
  next = x;
  for (int m = 0; m < M.l0; ++m) legendre_next(M, m, x, p, next);
}

__global__ void drop_kernel(DropMap M, double* rho) {
  const int n = blockIdx.x * blockDim.x + threadIdx.x;
  if (n >= M.Nz * M.Nr) return;
  const int j = n / M.Nz, k = n - j * M.Nz;
  const double dz = k - M.zc, r = j + 0.5, d = sqrt(dz * dz + r * r), ct = dz / d;
  double s = 0.0, p, next;
  legendre_start(M, ct, p, next);
  for (int m = 0; m < M.namp; ++m) {
    s += M.amp[m] * p;
    legendre_next(M, M.l0 + m, ct, p, next);
  }
  const double Rs = M.R * (1.0 + s);
  rho[n] = M.rho_v + 0.5 * (M.rho_l - M.rho_v) * (1.0 - tanh((d - Rs) / M.w));
}

constexpr int RED_NT = 256;
// per-block sums of sum_x rho_bar(x) d rho(x) / d a_m, rho_bar = sum_i W_i lambda^0_i;
// N >= namp amplitudes in registers
template <class C, int N>
__global__ void __launch_bounds__(RED_NT) drop_adj_kernel(DropMap M, const C* lam, size_t plane,
                                                          int P, double* partials) {
  __shared__ double red[RED_NT / 32][N];
  double acc[N];
#pragma unroll
  for (int m = 0; m < N; ++m) acc[m] = 0.0;
  for (int n = blockIdx.x * RED_NT + threadIdx.x; n < M.Nz * M.Nr; n += gridDim.x * RED_NT) {
    const int j = n / M.Nz, k = n - j * M.Nz;
    const size_t o = (size_t)j * P + k;
    double rb = 0.0;
#pragma unroll
    for (int q = 0; q < 9; ++q) rb += aw(q) * double(lam[q * plane + o]);
    const double dz = k - M.zc, r = j + 0.5, d = sqrt(dz * dz + r * r), ct = dz / d;
    double s = 0.0, p, next;
    legendre_start(M, ct, p, next);
    const double p0 = p, next0 = next;
    for (int m = 0; m < M.namp; ++m) {
      s += M.amp[m] * p;
      legendre_next(M, M.l0 + m, ct, p, next);
    }
    const double X = (d - M.R * (1.0 + s)) / M.w, sh = 1.0 / cosh(X);
    const double c = rb * (0.5 * (M.rho_l - M.rho_v) * sh * sh / M.w) * M.R;
    p = p0;
    next = next0;
#pragma unroll
    for (int m = 0; m < N; ++m) {
      if (m >= M.namp) break;
      acc[m] += c * p;
      legendre_next(M, M.l0 + m, ct, p, next);
    }
  }
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int m = 0; m < N; ++m) {
    if (m >= M.namp) break;
    double v = acc[m];
    for (int w = 16; w > 0; w >>= 1) v += __shfl_xor_sync(0xffffffffu, v, w);
    if (lane == 0) red[warp][m] = v;
  }
  __syncthreads();
  if ((int)threadIdx.x < M.namp) {
    double v = 0.0;
    for (int w = 0; w < RED_NT / 32; ++w) v += red[w][threadIdx.x];
    partials[blockIdx.x * 32 + threadIdx.x] = v;
  }
}

// per-block sums of two per-site FP64 arrays ([Nr][P]) -> partials[b * 2 + {0, 1}]
__global__ void __launch_bounds__(RED_NT) sum2_kernel(const double* a, const double* b, int Nz, int Nr,
                                                      int P, double* partials) {
  __shared__ double ra[RED_NT], rb[RED_NT];
  double sa = 0.0, sb = 0.0;
  for (int n = blockIdx.x * RED_NT + threadIdx.x; n < Nz * Nr; n += gridDim.x * RED_NT) {
    const int j = n / Nz, k = n - j * Nz;
    sa += a[(size_t)j * P + k];
    sb += b[(size_t)j * P + k];
  }
  ra[threadIdx.x] = sa;
  rb[threadIdx.x] = sb;
  __syncthreads();
  for (int s = RED_NT / 2; s > 0; s >>= 1) {
    if (threadIdx.x < s) {
      ra[threadIdx.x] += ra[threadIdx.x + s];
      rb[threadIdx.x] += rb[threadIdx.x + s];
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    partials[blockIdx.x * 2] = ra[0];
    partials[blockIdx.x * 2 + 1] = rb[0];
  }
}

// lambda^T = dJ/df_i(x) = dJ/drho(x) for every i; coef: the objective's constant factor
template <class C>
__global__ void seed_kernel(int kind, int Nz, int Nr, int P, size_t plane, double zc, int kstar, double coef, C* lam) {
  const int n = blockIdx.x * blockDim.x + threadIdx.x;
  if (n >= Nz * Nr) return;
  const int j = n / Nz, k = n - j * Nz;
  const double r = j + 0.5, dz = k - zc;
  const double s = kind == AMLBM_OBJ_A2SQ ? coef * (r * (dz * dz - 0.5 * r * r)) : k == kstar ? coef * r : 0.0;
#pragma unroll
  for (int q = 0; q < 9; ++q) lam[q * plane + (size_t)j * P + k] = C(s);
}

// J of the neck objective from the read-back density (one thread)
template <class C>
__global__ void neck_kernel(const C* rho, int Nz, int Nr, int kstar, double rho_l, double rho_v, double* J) {
  double s = 0.0;
  for (int j = 0; j < Nr; ++j) s += (j + 0.5) * (double(rho[(size_t)j * Nz + kstar]) - rho_v) / (rho_l - rho_v);
  *J = sqrt(2.0 * s);
}

}  // namespace
}  // namespace amlbm

// ------------------------------------------------------------------ driver --
using amlbm::InstDesc;

namespace {

struct AdjLayout {
  size_t total = 0;
  size_t ckpt = 0, seg = 0, lam = 0, inter = 0, fstar = 0, arr = 0, acc = 0, rho0 = 0,
         red = 0, descs = 0, tiles = 0;
  int nck = 0, nseg = 0, ntiles = 0, nred = 0;
  int nbuf = 1;            // segment buffers: two when there are several segments
  size_t state_elems = 0;  // 10 planes (f and psi)
};

constexpr int kAdjArrays = 9;

size_t al(size_t x) { return (x + 255) / 256 * 256; }

AdjLayout adj_layout(const amlbm::CtxInfo& ci, const amlbm_adjoint_problem& p) {
  AdjLayout L;
  const size_t cb = ci.storage == AMLBM_STORE_F64 ? 8 : 4;
  const size_t plane = (size_t)ci.host.P * ci.Nr;
  L.nck = (p.T + p.ckpt_every - 1) / p.ckpt_every;
  L.nseg = std::min(p.ckpt_every, p.T);
  L.nbuf = L.nck > 1 ? 2 : 1;
  L.state_elems = 10 * plane;
  int tz, tr;
  amlbm::inter_tile(ci.storage, ci.Nz, ci.Nr, &tz, &tr);
  L.ntiles = ((ci.Nz + tz - 1) / tz) * ((ci.Nr + tr - 1) / tr);
  L.nred = std::min(1024, (ci.Nz * ci.Nr + 255) / 256);
  size_t o = 0;
  auto take = [&](size_t b) { const size_t a = o; o = al(o + b); return a; };
  L.ckpt = take((size_t)L.nck * L.state_elems * cb);
  // per segment buffer: the segment's states and their intermediates
  L.seg = take((size_t)L.nbuf * (L.nseg + 1) * L.state_elems * cb);
  L.lam = take(2 * 9 * plane * cb);
  L.inter = take((size_t)L.nbuf * L.nseg * amlbm::I_COUNT * plane * cb);
  L.fstar = take(ci.storage == AMLBM_STORE_F64 ? 9 * plane * cb : 0);
  L.arr = take((size_t)kAdjArrays * plane * cb);
  L.acc = take(2 * plane * sizeof(double));
  L.rho0 = take((size_t)ci.Nz * ci.Nr * sizeof(double));
  const int nblk = amlbm::diag_blocks(ci.Nz, ci.Nr, (long long)ci.Nz * ci.Nr);
  L.red = take((size_t)(std::max(L.nred * 34, 8 * nblk + ci.Nz + 16) + 64) * sizeof(double));
  L.descs = take((size_t)L.nbuf * L.nseg * sizeof(InstDesc));
  L.tiles = take((size_t)L.ntiles * sizeof(int));
  L.total = o;
  return L;
}

int check_problem(const amlbm::CtxInfo& ci, const amlbm_adjoint_problem* p) {
  using amlbm::set_error;
  if (!p) return set_error(AMLBM_EINVAL, "NULL problem");
  if (ci.storage != AMLBM_STORE_F64 && ci.storage != AMLBM_STORE_F32)
    return set_error(AMLBM_EINVAL, "the adjoint needs FP64 or FP32 storage");
  if (ci.host.shift != 0) return set_error(AMLBM_EINVAL, "the adjoint needs unshifted storage");
  if (ci.host.zbc != AMLBM_Z_PERIODIC || ci.host.rlo != AMLBM_RLO_AXIS || ci.host.wall == AMLBM_WALL_OUTLET)
    return set_error(AMLBM_EINVAL, "the adjoint takes periodic lattices on the axis only");
  if (ci.host.forcing != AMLBM_FORCE_SHIFT)
    return set_error(AMLBM_EINVAL, "the adjoint implements the velocity-shift forcing only");
  if (ci.host.src != AMLBM_SRC_LOCAL)
    return set_error(AMLBM_EINVAL, "the adjoint implements the departure-site source only");
  if (p->T < 1 || p->ckpt_every < 1) return set_error(AMLBM_EINVAL, "need T >= 1, ckpt_every >= 1");
  if (p->n_amps < 0 || p->n_amps > 32 || (p->n_amps > 0 && !p->amps) || p->l0 < 0)
    return set_error(AMLBM_EINVAL, "need 0 <= n_amps <= 32, amps, l0 >= 0");
  if (p->objective != AMLBM_OBJ_A2SQ && p->objective != AMLBM_OBJ_NECK)
    return set_error(AMLBM_EINVAL, "bad objective");
  if (p->objective == AMLBM_OBJ_NECK && (p->kstar < 0 || p->kstar >= ci.Nz))
    return set_error(AMLBM_EINVAL, "kstar outside the lattice");
  if (!(p->w > 0) || !(p->R > 0) || !(p->obj_R > 0) || !(p->rho_l != p->rho_v))
    return set_error(AMLBM_EINVAL, "need w > 0, R > 0, obj_R > 0, rho_l != rho_v");
  return AMLBM_OK;
}

#define ADJ_CK(call)                                                                   \
  do {                                                                                 \
    cudaError_t e_ = (call);                                                           \
    if (e_ != cudaSuccess) {                                                           \
      rc = amlbm::set_error(AMLBM_ECUDA, std::string(#call) + ": " + cudaGetErrorString(e_)); \
      goto done;                                                                       \
    }                                                                                  \
  } while (0)

template <class C>
int run(amlbm_ctx* ctx, const amlbm_adjoint_problem* p, void* ws, size_t ws_bytes, bool adjoint,
        double* J, double* dG, double* dT, double* dA) {
  using namespace amlbm;
  CtxInfo ci;
  int rc = ctx_info(ctx, &ci);
  if (rc) return rc;
  if ((rc = check_problem(ci, p))) return rc;
  const AdjLayout L = adj_layout(ci, *p);
  const cudaStream_t s = ci.stream;
  const int Nz = ci.Nz, Nr = ci.Nr, P = ci.host.P, N = Nz * Nr;
  const size_t plane = (size_t)P * Nr;
  const int nb = (N + 255) / 256;
  char* base = static_cast<char*>(ws);
  bool owns = false;
  std::vector<double> red;
  double Jv = 0.0;
  if (!base) {
    const cudaError_t e = cudaMalloc(&base, L.total);
    if (e != cudaSuccess) return set_error(AMLBM_ENOMEM, std::string("cudaMalloc: ") + cudaGetErrorString(e));
    owns = true;
  } else if (ws_bytes < L.total || reinterpret_cast<uintptr_t>(ws) % 256) {
    return set_error(AMLBM_ENOMEM, "adjoint workspace too small or not 256-byte aligned: need " +
                                       std::to_string(L.total) + " bytes");
  }
  {
    C* ckpt = reinterpret_cast<C*>(base + L.ckpt);
    C* seg = reinterpret_cast<C*>(base + L.seg);
    C* lam[2] = {reinterpret_cast<C*>(base + L.lam), reinterpret_cast<C*>(base + L.lam) + 9 * plane};
    double* rho_init = reinterpret_cast<double*>(base + L.rho0);
    double* redbuf = reinterpret_cast<double*>(base + L.red);
    const size_t SB = L.state_elems * sizeof(C), FB = 9 * plane * sizeof(C), PB = plane * sizeof(C);
    void* fcur;
    void* pcur;
    int pitch, tz, tr;

    DropMap M;
    std::memset(&M, 0, sizeof(M));
    M.Nz = Nz; M.Nr = Nr; M.l0 = p->l0; M.namp = p->n_amps;
    M.zc = p->zc; M.R = p->R; M.w = p->w; M.rho_l = p->rho_l; M.rho_v = p->rho_v;
    for (int m = 0; m < p->n_amps; ++m) M.amp[m] = p->amps[m];
    for (int m = 1; m < kMaxDegree; ++m) M.inv[m] = 1.0 / m;

    // forward: initial drop, T steps, states every ckpt_every steps
    drop_kernel<<<nb, 256, 0, s>>>(M, rho_init);
    ADJ_CK(cudaGetLastError());
    ADJ_CK(launch_init(ci.storage, ci.d_desc, 0, Nz, Nr, rho_init, nullptr, nullptr, ci.parity, s));
    for (int n = 0; n < p->T; ++n) {
      if (adjoint && n % p->ckpt_every == 0) {
        amlbm_device_state(ctx, &fcur, &pcur, &pitch);
        C* dst = ckpt + (size_t)(n / p->ckpt_every) * L.state_elems;
        ADJ_CK(cudaMemcpyAsync(dst, fcur, FB, cudaMemcpyDeviceToDevice, s));
        ADJ_CK(cudaMemcpyAsync(dst + 9 * plane, pcur, PB, cudaMemcpyDeviceToDevice, s));
      }
      if ((rc = amlbm_step(ctx, 1))) goto done;
    }
    // objective of the final state
    if ((rc = ctx_readback(ctx))) goto done;
    {
      double a2 = 0.0;
      if (p->objective == AMLBM_OBJ_A2SQ) {
        const int nblk = diag_blocks(Nz, Nr, (long long)Nz * Nr);
        ADJ_CK(launch_diag(ci.storage, ci.d_desc, 0, Nz, Nr, ci.parity ^ (p->T & 1), p->zc, p->obj_R,
                           p->rho_l, p->rho_v, redbuf, nblk, redbuf + 8 * nblk, redbuf + 8 * nblk + Nz, s));
        ADJ_CK(cudaMemcpyAsync(&a2, redbuf + 8 * nblk + Nz + 5, sizeof(double), cudaMemcpyDeviceToHost, s));
        ADJ_CK(cudaStreamSynchronize(s));
        Jv = a2 * a2;
      } else {
        neck_kernel<C><<<1, 1, 0, s>>>(static_cast<const C*>(ci.host.rho_out), Nz, Nr, p->kstar, p->rho_l,
                                       p->rho_v, redbuf);
        ADJ_CK(cudaGetLastError());
        ADJ_CK(cudaMemcpyAsync(&Jv, redbuf, sizeof(double), cudaMemcpyDeviceToHost, s));
        ADJ_CK(cudaStreamSynchronize(s));
      }
      if (J) *J = Jv;
      if (!adjoint) goto done;
      // J = a2^2, a2 = a2_norm sum 2 pi r phi (dz^2 - r^2/2); or J = sqrt(2 sum r phi)
      const double coef = p->objective == AMLBM_OBJ_A2SQ
                              ? 2.0 * a2 * a2_norm(p->obj_R) * 2.0 * 3.14159265358979323846 / (p->rho_l - p->rho_v)
                              : 1.0 / ((p->rho_l - p->rho_v) * Jv);
      seed_kernel<C><<<nb, 256, 0, s>>>(p->objective, Nz, Nr, P, plane, p->zc, p->kstar, coef, lam[0]);
      ADJ_CK(cudaGetLastError());
    }
    // descriptors of the segment slots (tiled by inter_tile): descriptor q of buffer b
    // steps slot q of that buffer into slot q + 1
    {
      std::vector<InstDesc> d((size_t)L.nbuf * L.nseg, ci.host);
      inter_tile(ci.storage, Nz, Nr, &tz, &tr);
      for (int b = 0; b < L.nbuf; ++b)
        for (int q = 0; q < L.nseg; ++q) {
          InstDesc& x = d[(size_t)b * L.nseg + q];
          x.tiles_z = (Nz + tz - 1) / tz;
          x.tiles_r = (Nr + tr - 1) / tr;
          x.tile_base = 0;
          C* sb = seg + (size_t)b * (L.nseg + 1) * L.state_elems;
          for (int h = 0; h < 2; ++h) {
            x.f[h] = sb + (size_t)(q + h) * L.state_elems;
            x.psi[h] = sb + (size_t)(q + h) * L.state_elems + 9 * plane;
          }
        }
      std::vector<int> tiles(L.ntiles, 0);
      ADJ_CK(cudaMemcpyAsync(base + L.descs, d.data(), d.size() * sizeof(InstDesc), cudaMemcpyHostToDevice, s));
      ADJ_CK(cudaMemcpyAsync(base + L.tiles, tiles.data(), tiles.size() * sizeof(int), cudaMemcpyHostToDevice, s));
      ADJ_CK(cudaMemsetAsync(base + L.acc, 0, 2 * plane * sizeof(double), s));
      ADJ_CK(cudaStreamSynchronize(s));  // host vectors above go out of scope
    }
    {
      Adj<C> A;
      A.Nz = Nz; A.Nr = Nr; A.P = P; A.wall = ci.host.wall; A.axisym = ci.host.axisym;
      A.plane = plane;
      A.tau = C(ci.host.tau); A.omega = C(1) / A.tau; A.G = C(ci.host.G);
      A.gz = C(ci.host.gz);
      A.inv_rho0 = C(1.0 / ci.host.rho0);
      C* arr = reinterpret_cast<C*>(base + L.arr);
      C** fields[kAdjArrays] = {&A.rhob, &A.jzb, &A.jrb, &A.psib, &A.qz, &A.qr, &A.dzrb, &A.drrb, &A.drdb};
      for (int q = 0; q < kAdjArrays; ++q) *fields[q] = arr + (size_t)q * plane;
      A.accG = reinterpret_cast<double*>(base + L.acc);
      A.accT = A.accG + plane;
      const InstDesc* d_seg = reinterpret_cast<const InstDesc*>(base + L.descs);
      const int* d_tiles = reinterpret_cast<const int*>(base + L.tiles);
      // 32 x 8 tiles, or 32 x 4 where those would leave SMs without one
      const int gz = (Nz + ATZ - 1) / ATZ;
      const bool low = gz * ((Nr + 7) / 8) < 152;
      C* inter_seg = reinterpret_cast<C*>(base + L.inter);
      const size_t iseg = (size_t)I_COUNT * plane;
      // Segment buffer b: states, intermediates and step descriptors.
      auto seg_of = [&](int b) { return seg + (size_t)b * (L.nseg + 1) * L.state_elems; };
      auto inter_of = [&](int b) { return inter_seg + (size_t)b * L.nseg * iseg; };
      // The recompute of a segment of `len` steps into buffer b (each step writes
      // the next state and the intermediates of the state it starts from).
      auto recompute = [&](int len, int b, cudaStream_t st) -> cudaError_t {
        for (int q = 0; q < len; ++q) {
          const cudaError_t e = launch_step_inter(ci.storage, tz, tr, d_seg + (size_t)b * L.nseg + q, d_tiles, L.ntiles,
                                                  inter_of(b) + q * iseg, plane, base + L.fstar, st);
          if (e != cudaSuccess) return e;
        }
        return cudaSuccess;
      };
      // The transposed steps of a segment in buffer b, from the last to the first,
      // starting with lambda in lam[c0].
      auto backward = [&](int len, int b, int c0, cudaStream_t st) -> cudaError_t {
        Adj<C> B = A;
        int c = c0;
        for (int q = len - 1; q >= 0; --q) {
          B.inter = inter_of(b) + q * iseg;
          B.f = seg_of(b) + (size_t)q * L.state_elems;
          B.lam_in = lam[c];
          B.lam_out = lam[c ^ 1];
          const dim3 grid(gz, low ? (Nr + 3) / 4 : (Nr + 7) / 8);
          cudaError_t e = low ? launch_pdl(adj_local<C, 4>, grid, ATZ * 4, 0, st, B)
                              : launch_pdl(adj_local<C, 8>, grid, ATZ * 8, 0, st, B);
          if (e == cudaSuccess)
            e = low ? launch_pdl(adj_psi<C, 4>, grid, ATZ * 4, 0, st, B)
                    : launch_pdl(adj_psi<C, 8>, grid, ATZ * 8, 0, st, B);
          if (e != cudaSuccess) return e;
          c ^= 1;
        }
        return cudaSuccess;
      };
      // Segments run from the last to the first.  The recompute of segment m - 1
      // (on stream rs, into the other buffer) does not depend on the backward
      // sweep of segment m (on s), so the two overlap: each is a few hundred CTAs
      // and leaves most of the GPU idle.  Events order each recompute after the
      // backward sweep that last read its buffer, and each backward sweep after
      // its recompute.  (The host issues the four launches of a step, three in FP32, faster
      // than the GPU runs them; capturing each call's segments into graphs cost more than
      // it saved.)
      cudaStream_t rs = nullptr;
      cudaEvent_t ev0 = nullptr, evR[2] = {nullptr, nullptr}, evB[2] = {nullptr, nullptr};
      bool usedB[2] = {false, false};
      bool streams_ok = cudaStreamCreateWithFlags(&rs, cudaStreamNonBlocking) == cudaSuccess &&
                        cudaEventCreateWithFlags(&ev0, cudaEventDisableTiming) == cudaSuccess;
      for (int b = 0; b < 2 && streams_ok; ++b)
        streams_ok = cudaEventCreateWithFlags(&evR[b], cudaEventDisableTiming) == cudaSuccess &&
                     cudaEventCreateWithFlags(&evB[b], cudaEventDisableTiming) == cudaSuccess;
      cudaStream_t rstream = streams_ok ? rs : s;  // without a second stream, no overlap
#define SEG_CK(call)                                                                          \
  {                                                                                           \
    const cudaError_t e_ = (call);                                                            \
    if (e_ != cudaSuccess) {                                                                  \
      rc = amlbm::set_error(AMLBM_ECUDA, std::string(#call) + ": " + cudaGetErrorString(e_)); \
      break;                                                                                  \
    }                                                                                         \
  }
      // issue the checkpoint copy and the recompute of segment m into buffer b on rstream
      auto issue_recompute = [&](int m, int b) -> cudaError_t {
        const int n0 = m * p->ckpt_every, len = std::min(p->T, n0 + p->ckpt_every) - n0;
        if (streams_ok && usedB[b]) {  // the backward sweep that last read buffer b
          const cudaError_t e = cudaStreamWaitEvent(rstream, evB[b], 0);
          if (e != cudaSuccess) return e;
        }
        cudaError_t e = cudaMemcpyAsync(seg_of(b), ckpt + (size_t)m * L.state_elems, SB,
                                        cudaMemcpyDeviceToDevice, rstream);
        if (e != cudaSuccess) return e;
        e = recompute(len, b, rstream);
        if (e == cudaSuccess && streams_ok) e = cudaEventRecord(evR[b], rstream);
        return e;
      };
      int cur = 0;
      do {
        if (streams_ok) {  // the recompute stream starts after the forward run and the seed
          SEG_CK(cudaEventRecord(ev0, s));
          SEG_CK(cudaStreamWaitEvent(rs, ev0, 0));
        }
        SEG_CK(issue_recompute(L.nck - 1, (L.nck - 1) % L.nbuf));
        for (int m = L.nck - 1; m >= 0 && rc == AMLBM_OK; --m) {
          const int b = m % L.nbuf;
          const int n0 = m * p->ckpt_every, len = std::min(p->T, n0 + p->ckpt_every) - n0;
          // the next segment's recompute goes ahead on the other buffer; with one
          // stream it would have to wait for this backward sweep, so it is issued after it
          if (m >= 1 && streams_ok) SEG_CK(issue_recompute(m - 1, (m - 1) % L.nbuf));
          if (streams_ok) SEG_CK(cudaStreamWaitEvent(s, evR[b], 0));
          SEG_CK(backward(len, b, cur, s));
          if (streams_ok) {
            SEG_CK(cudaEventRecord(evB[b], s));
            usedB[b] = true;
          }
          if (m >= 1 && !streams_ok) SEG_CK(issue_recompute(m - 1, (m - 1) % L.nbuf));
          if (len & 1) cur ^= 1;
        }
      } while (false);
      if (rs) cudaStreamSynchronize(rs);
      cudaStreamSynchronize(s);
      for (auto* ev : {ev0, evR[0], evR[1], evB[0], evB[1]})
        if (ev) cudaEventDestroy(ev);
      if (rs) cudaStreamDestroy(rs);
#undef SEG_CK
      if (rc) goto done;
      // parameter gradients (FP64, fixed order)
      sum2_kernel<<<L.nred, RED_NT, 0, s>>>(A.accG, A.accT, Nz, Nr, P, redbuf);
      ADJ_CK(cudaGetLastError());
      if (p->n_amps > 0) {
        double* part = redbuf + 2 * L.nred;
        if (p->n_amps <= 4) drop_adj_kernel<C, 4><<<L.nred, RED_NT, 0, s>>>(M, lam[cur], plane, P, part);
        else if (p->n_amps <= 16) drop_adj_kernel<C, 16><<<L.nred, RED_NT, 0, s>>>(M, lam[cur], plane, P, part);
        else drop_adj_kernel<C, 32><<<L.nred, RED_NT, 0, s>>>(M, lam[cur], plane, P, part);
        ADJ_CK(cudaGetLastError());
      }
      red.resize((size_t)L.nred * 34);
      ADJ_CK(cudaMemcpyAsync(red.data(), redbuf, red.size() * sizeof(double), cudaMemcpyDeviceToHost, s));
      ADJ_CK(cudaStreamSynchronize(s));
      double g = 0.0, t = 0.0;
      for (int b = 0; b < L.nred; ++b) { g += red[2 * b]; t += red[2 * b + 1]; }
      if (dG) *dG = g;
      if (dT) *dT = t;
      for (int m = 0; m < p->n_amps; ++m) {
        double a = 0.0;
        for (int b = 0; b < L.nred; ++b) a += red[2 * L.nred + (size_t)b * 32 + m];
        if (dA) dA[m] = a;
      }
    }
  }
done:
  if (owns) {
    cudaStreamSynchronize(s);
    cudaFree(base);
  }
  return rc;
}

}  // namespace

extern "C" {

size_t amlbm_adjoint_workspace_bytes(amlbm_ctx* ctx, const amlbm_adjoint_problem* p) {
  amlbm::CtxInfo ci;
  if (!ctx || amlbm::ctx_info(ctx, &ci) || check_problem(ci, p)) return 0;
  return adj_layout(ci, *p).total;
}

int amlbm_adjoint(amlbm_ctx* ctx, const amlbm_adjoint_problem* p, void* workspace, size_t bytes,
                  double* J, double* dJ_dG, double* dJ_dtau, double* dJ_damps) {
  amlbm::CtxInfo ci;
  if (!ctx) return amlbm::set_error(AMLBM_EINVAL, "NULL context");
  const int rc = amlbm::ctx_info(ctx, &ci);
  if (rc) return rc;
  if (ci.storage == AMLBM_STORE_F64)
    return run<double>(ctx, p, workspace, bytes, true, J, dJ_dG, dJ_dtau, dJ_damps);
  return run<float>(ctx, p, workspace, bytes, true, J, dJ_dG, dJ_dtau, dJ_damps);
}

int amlbm_objective(amlbm_ctx* ctx, const amlbm_adjoint_problem* p, double* J) {
  amlbm::CtxInfo ci;
  if (!ctx) return amlbm::set_error(AMLBM_EINVAL, "NULL context");
  const int rc = amlbm::ctx_info(ctx, &ci);
  if (rc) return rc;
  if (ci.storage == AMLBM_STORE_F64) return run<double>(ctx, p, nullptr, 0, false, J, nullptr, nullptr, nullptr);
  return run<float>(ctx, p, nullptr, 0, false, J, nullptr, nullptr, nullptr);
}

}  // extern "C"
