// The FP64 form's two-kernel step for sm_103a (arXiv:1310.1871, Sec. II).
//
// GB300 issues one FP64 warp instruction per 16.4 clocks and SM (measured), so the
// FP64 step is bound by the number of FP64 operations, and on small lattices by how
// many SMs share them; memory and instruction issue are idle beside that.  The two
// kernels evaluate nearly every operation once per site, with no recomputed halo
// but d_r psi (tile + 2) and the sources (tile + 1):
//
//   f64_force  : psi (tile + 4) -> isotropic d_r psi (tile + 2), 1D d_r psi -> F_SC
//                (Eq. scforce), F^gamma (Eq. scAxisExtra), body force; moments, u; the
//                BGK collision (Eq. lbm2d) of the site, written over the site's own
//                populations (nothing reads them again); u_z, u_r and rho into planes
//   f64_stream : u (tile + 3) with its ghost rules -> velocity gradients -> S, H_z, H_r
//                (Eq. condition_h) on the tile + 1; then every site pulls the nine
//                collided populations (axis, wall, periodic and bounce-back maps of
//                Sec. II.E) with the sources of their departure sites, and psi of the
//                new state
//
// 214 FP64 operations per site (exp counts 20) on 32 x 8 tiles, against 472 for the
// kernels that recomputed the collision on the streaming halo.  The arithmetic is
// that of every other FP64 schedule, operation for operation, so the states are
// bit-identical.  It takes every lattice the fused schedule takes.
//
// On small grids each kernel lets the next start as soon as it has begun to read
// (pdl_trigger): its blocks then wait beside this one's with their index and row
// constants ready.  us per step without / with it: 64 x 32 (64 blocks of 8 x 4) 10.8 / 8.9,
// 128 x 64 (256) 13.2 / 11.5, 192 x 80 (480) 17.8 / 16.6, 256 x 128 (128 of 32 x 8) 23.1 / 21.4,
// 384 x 200 (300) 38.0 / 36.8.  Beyond, the next kernel's blocks crowd onto the SMs that are
// free first: 192 x 120 (180 of 16 x 8) 23.6 / 27.3, 512 x 200 (400 of 32 x 8) 52.2 / 65.7.  The
// adjoint's forward steps (MODE 3) never do: they run beside another stream, whose kernels
// need the room (gradient of 256 x 128 over 50 steps 3.77 ms, with it 4.15).
// The figures for every tile stand beside pick_tile (amlbm_abi.cu), which chooses it.

#include <stdint.h>

#include <type_traits>

#include "amlbm.h"
#include "amlbm_internal.cuh"
#include "amlbm_launch.cuh"
#include "amlbm_physics.cuh"

namespace amlbm {
namespace {

// Tile geometry and threads.  An FP64 warp instruction occupies its SM sub-partition's
// FP64 unit for 64 clocks, so a lattice of few sites is bound by the length of one
// site's chain of operations, not by throughput: tiles of fewer than 256 sites take
// ROLES threads per site, each with a share of the force and moment terms and of the
// nine directions (the values they share go through shared memory).  The terms needed
// by every share (u, u^eq) are evaluated by each, so large lattices, which are bound by
// throughput, take one thread per site.
template <int BZ, int BR>
struct Geo64 {
  static constexpr int SITES = BZ * BR;
  static constexpr int ROLES = SITES >= 256 ? 1 : SITES >= 128 ? 2 : 4;
  static constexpr int NT = SITES * ROLES < 256 ? SITES * ROLES : 256;
  static_assert(SITES % 32 == 0 && (ROLES == 1 || NT == SITES * ROLES), "a role is whole warps");
  // CTAs of f64_force per SM that its registers have to allow: on 512-site tiles three (79
  // registers; left to itself the compiler takes 94).  On 256-site tiles it takes 64 by
  // itself, which the early launch below needs: two CTAs of this kernel and two of the
  // next fit an SM then.  With the nine populations held until the last is formed it takes
  // 78, and 384 x 200 took 58.2 us a step, 304 x 160 45.7 (36.8 and 36.2).
  static constexpr int kBlocks = SITES > 256 ? 3 : 0;
  // the largest grid that starts the next kernel early
  static constexpr unsigned kEarly = ROLES == 4 ? 512 : SITES == 256 ? 304 : 152;
  static constexpr int PZ = BZ + 8, PR = BR + 8;  // psi
  static constexpr int DZ = BZ + 4, DR = BR + 4;  // isotropic d_r psi
  static constexpr int FZ = BZ + 6, FR = BR + 6;  // u
  static constexpr int SZ = BZ + 2, SR = BR + 2;  // sources
};

template <int NT, int ROWS, int W, class F>
__device__ __forceinline__ void for_sites(F&& body) {
  for (int t = threadIdx.x; t < ROWS * W; t += NT) {
    const int lr = t / W;
    body(lr, t - lr * W);
  }
}

// The role that handles direction i: pairs of opposite directions stay together (they
// share their parts).  The rest population, which takes what the pairs leave of rho, comes
// last, from the role of the first pair.
__host__ __device__ constexpr int pair_of(int i) {
  return i == 0 || i == 1 || i == 3 ? 0 : i == 2 || i == 4 ? 1 : i == 5 || i == 7 ? 2 : 3;
}
__host__ __device__ constexpr int role_of(int i, int roles) { return pair_of(i) % roles; }

// In f64_stream the directions are split by the terms of moment0, of which each role adds
// its own (64 x 32: 0.2 us per step): part p, of role p % roles.
__host__ __device__ constexpr int part_of(int i) {
  return i == 0 || i == 2 || i == 4 ? 0 : i == 1 || i == 3 ? 1 : i == 5 || i == 6 ? 2 : 3;
}
__host__ __device__ constexpr int pull_role(int i, int roles) { return part_of(i) % roles; }

// body(integral_constant role) for this thread's role (uniform in a warp)
template <int ROLES, class F>
__device__ __forceinline__ void with_role(int role, F&& body) {
  if constexpr (ROLES == 1) {
    body(std::integral_constant<int, 0>());
  } else {
    switch (role) {
      case 0: body(std::integral_constant<int, 0>()); break;
      case 1: body(std::integral_constant<int, 1>()); break;
      case 2: if constexpr (ROLES > 2) body(std::integral_constant<int, 2>()); break;
      default: if constexpr (ROLES > 2) body(std::integral_constant<int, 3>()); break;
    }
  }
}

// MODE 0: the step's first half; MODE 1: rho and u into the read-back planes (the
// state is left alone); MODE 3: the step's first half with the forward intermediates
// for the adjoint (into `inter`), the collided populations going to `fstar`.
template <int BZ, int BR, int MODE>
__global__ void __launch_bounds__(Geo64<BZ, BR>::NT, MODE == 0 ? Geo64<BZ, BR>::kBlocks : 0) f64_force(const InstDesc* __restrict__ descs,
                                                              const int* __restrict__ tile_inst, int toff,
                                                              int parity, double* __restrict__ inter, size_t iplane,
                                                              double* fstar) {
  using T = D1;
  using G = Geo64<BZ, BR>;
  constexpr int ROLES = G::ROLES;
  __shared__ T sPsi[G::PR * G::PZ], sDr[G::DR * G::DZ], sD1[BR * G::DZ];
  __shared__ T sX[ROLES > 1 ? 14 * G::SITES : 1];  // what the roles of a site share
  __shared__ Row<T> sRow[BR];
  __shared__ int sCol[G::PZ], sOff[G::PR];
  const int tile = blockIdx.x + toff;
  const InstDesc& D = descs[tile_inst[tile]];
  const int Nz = D.Nz, Nr = D.Nr, P = D.P;
  const int l = tile - (MODE == 1 ? D.rb_tile_base : D.tile_base);
  const int tz = MODE == 1 ? D.rb_tiles_z : D.tiles_z;
  const int k0 = (l % tz) * BZ, j0 = (l / tz) * BR;
  const size_t plane = (size_t)P * Nr;
  double* f = static_cast<double*>(D.f[parity]);
  const double* psin = static_cast<const double*>(D.psi[parity]);
  const bool ax = D.axisym != 0, zw = D.zbc == AMLBM_Z_NOSLIP;
  const bool inl = D.rlo == AMLBM_RLO_INLET, outl = D.wall == AMLBM_WALL_OUTLET;
  const bool guo = D.forcing == AMLBM_FORCE_GUO;
  const Par<T> q = par_of<T>(D);
  const T gk{D.k64[K_GUO]};
  for (int i = threadIdx.x; i < G::PZ; i += G::NT) sCol[i] = ghost_col(k0 - 4 + i, Nz, zw);
  for (int i = threadIdx.x; i < G::PR; i += G::NT) sOff[i] = ghost_row(j0 - 4 + i, Nr, inl, outl) * P;
  if (threadIdx.x < BR) sRow[threadIdx.x] = row_of(q, j0 + (int)threadIdx.x, D.k64[K_R0]);
  __syncthreads();
  pdl_wait();  // everything above reads only what creation wrote
  if (MODE != 3 && gridDim.x <= G::kEarly) pdl_trigger();

  for_sites<G::NT, G::PR, G::PZ>([&](int lr, int lc) { sPsi[lr * G::PZ + lc] = T{psin[sOff[lr] + sCol[lc]]}; });
  __syncthreads();
  if (ax) {
    for_sites<G::NT, G::DR, G::DZ>([&](int lr, int lc) {
      const T* p = sPsi + (lr + 2) * G::PZ + (lc + 2);
      sDr[lr * G::DZ + lc] = iso_r(p, G::PZ);
      if (lr >= 2 && lr < BR + 2) sD1[(lr - 2) * G::DZ + lc] = d1(p, G::PZ);
    });
    __syncthreads();
  }

  const int role = ROLES > 1 ? (int)threadIdx.x / G::SITES : 0;
  for (int t = (int)threadIdx.x - role * G::SITES; t < G::SITES; t += (ROLES > 1 ? G::SITES : G::NT)) {
    const int lr = t / BZ, lc = t - lr * BZ, j = j0 + lr, k = k0 + lc;
    const bool in = j < Nr && k < Nz;
    const size_t o = (size_t)(in ? j : 0) * P + (in ? k : 0);
    const T* p = sPsi + (lr + 4) * G::PZ + (lc + 4);
    const T* dr = sDr + (lr + 2) * G::DZ + (lc + 2);
    const T psi = p[0];
    const Row<T>& row = sRow[lr];
    double* out = (MODE == 3 ? fstar : f) + o;
    T fv[9], sz, sr, dr0 = lit<T>(0.0), Drr = lit<T>(0.0), Dzr = lit<T>(0.0), rho, jz, jr, inv_rho, Fz, Fr;
    if constexpr (ROLES == 1) {
      if (!in) continue;
#pragma unroll
      for (int i = 0; i < 9; ++i) fv[i] = T{f[i * plane + o]};
      sc_sums(p, G::PZ, sz, sr);
      if (ax) {
        dr0 = dr[0];
        Drr = iso_r(dr, G::DZ);
        Dzr = d1(sD1 + lr * G::DZ + (lc + 2), 1);
      }
      rho = moment0(fv);
      jz = moment_z(fv);
      jr = moment_r(fv);
      forces(q, rho, psi, sz, sr, ax, dr0, Drr, Dzr, row, Fz, Fr);
      inv_rho = rcp(rho);
    } else {
      // the terms of forces() and the moments, each from one role
      constexpr int NS = G::SITES;
      T* x = sX + t;
#pragma unroll
      for (int i = 0; i < 9; ++i) fv[i] = in ? T{f[i * plane + o]} : lit<T>(0.0);
      if (role == 0) {
        sc_sums(p, G::PZ, sz, sr);
        const T gpsi = psi * q.negG36;
        x[0] = gpsi * sz;
        x[NS] = gpsi * sr;
      }
      if (role == 1 && ax) {
        dr0 = dr[0];
        Drr = iso_r(dr, G::DZ);
        Dzr = d1(sD1 + lr * G::DZ + (lc + 2), 1);
        x[2 * NS] = psi * row.g9;
        x[3 * NS] = Dzr;
        x[4 * NS] = psi * row.g;
        x[5 * NS] = fma(-dr0, row.inv36, Drr);
      }
      if (role == 2 % ROLES) {
        const T m = moment0(fv);
        x[6 * NS] = m;
        x[7 * NS] = rcp(m);
      }
      if (role == 3 % ROLES) {
        x[8 * NS] = moment_z(fv);
        x[9 * NS] = moment_r(fv);
      }
      __syncthreads();
      rho = x[6 * NS];
      inv_rho = x[7 * NS];
      jz = x[8 * NS];
      jr = x[9 * NS];
      Fz = x[0];
      Fr = x[NS];
      if (ax) {
        Fz = fma(x[2 * NS], x[3 * NS], Fz);
        Fr = fma(x[4 * NS], x[5 * NS], Fr);
      }
      Fz = fma(rho, q.gz, Fz);
    }
    if (in) {
      const T uz = fma(Fz, lit<T>(0.5), jz) * inv_rho, ur = fma(Fr, lit<T>(0.5), jr) * inv_rho;
      if constexpr (MODE == 1) {
        const size_t w = (size_t)j * Nz + k;
        if (role == 0) {
          static_cast<double*>(D.rho_out)[w] = rho.v;
          static_cast<double*>(D.uz_out)[w] = uz.v;
          static_cast<double*>(D.ur_out)[w] = ur.v;
        }
      } else {
        if (role == ROLES - 1) {
          double* uv = static_cast<double*>(D.uv) + o;
          uv[0] = uz.v;
          uv[plane] = ur.v;
          uv[2 * plane] = rho.v;
        }
        if constexpr (MODE == 3) {
          double* w = inter + o;
          if (role == 0) {
            w[I_SZ * iplane] = unscale(sz, 36.0).v;
            w[I_SR * iplane] = unscale(sr, 36.0).v;
            w[I_PSI * iplane] = psi.v;
          }
          if (role == 1 % ROLES) {
            w[I_DR * iplane] = unscale(dr0, 36.0).v;
            w[I_DRR * iplane] = unscale(Drr, 1296.0).v;
            w[I_DZR * iplane] = unscale(Dzr, 144.0).v;
          }
          if (role == 2 % ROLES) {
            w[I_RHO * iplane] = rho.v;
            w[I_UZ * iplane] = uz.v;
            w[I_UR * iplane] = ur.v;
          }
          if (role == 3 % ROLES) {
            w[I_VZ * iplane] = (fma(Fz, q.tau, jz) * inv_rho).v;
            w[I_VR * iplane] = (fma(Fr, q.tau, jr) * inv_rho).v;
            w[I_FZ * iplane] = Fz.v;
            w[I_FR * iplane] = Fr.v;
          }
        }
        with_role<ROLES>(role, [&](auto R) {
          T g[9];
          collide(q, guo, gk, fv, rho, uz, ur, jz, jr, Fz, Fr, inv_rho, [&](int i, T v) {
            if (role_of(i, ROLES) != R.value || (ROLES > 1 && i == 0)) return;
            out[i * plane] = v.v;
            g[i] = v;
          });
          if constexpr (ROLES > 1) {  // the sums that leave the rest population
            constexpr int first[4] = {1, 2, 5, 6};
#pragma unroll
            for (int p = 0; p < 4; ++p)
              if (p % ROLES == R.value) sX[(10 + p) * G::SITES + t] = g[first[p]] + g[first[p] + 2];
          }
        });
      }
    }
    if constexpr (ROLES > 1 && MODE != 1) {
      __syncthreads();
      const T* x = sX + 10 * G::SITES + t;
      if (in && role == 0) out[0] = rest_of(rho, x[0], x[G::SITES], x[2 * G::SITES], x[3 * G::SITES]).v;
    }
  }
}

// MODE 0: the step's second half; MODE 3: with the velocity gradients for the adjoint.
template <int BZ, int BR, int MODE>
__global__ void __launch_bounds__(Geo64<BZ, BR>::NT) f64_stream(const InstDesc* __restrict__ descs,
                                                               const int* __restrict__ tile_inst, int parity,
                                                               double* __restrict__ inter, size_t iplane,
                                                               const double* fstar,
                                                               int* __restrict__ ctr) {
  using T = D1;
  using G = Geo64<BZ, BR>;
  constexpr int ROLES = G::ROLES;
  __shared__ T sUz[G::FR * G::FZ], sUr[G::FR * G::FZ];
  __shared__ T sS[G::SR * G::SZ], sHz[G::SR * G::SZ], sHr[G::SR * G::SZ];
  __shared__ T sB[2][9][G::SZ];  // populations of an inlet row and an outlet row
  __shared__ T sF[ROLES > 1 ? 4 * G::SITES : 1];  // the parts of rho
  __shared__ Row<T> sRow[G::SR];
  __shared__ int sCol[G::FZ];
  const int tile = blockIdx.x;
  const InstDesc& D = descs[tile_inst[tile]];
  const int Nz = D.Nz, Nr = D.Nr, P = D.P;
  const int l = tile - D.tile_base;
  const int k0 = (l % D.tiles_z) * BZ, j0 = (l / D.tiles_z) * BR;
  const size_t plane = (size_t)P * Nr;
  const double* fs = MODE == 3 ? fstar : static_cast<const double*>(D.f[parity]);
  const double* uv = static_cast<const double*>(D.uv);
  const bool ax = D.axisym != 0, zw = D.zbc == AMLBM_Z_NOSLIP;
  const bool inl = D.rlo == AMLBM_RLO_INLET, outl = D.wall == AMLBM_WALL_OUTLET;
  const bool noslip = D.wall == AMLBM_WALL_NOSLIP, link = D.src == AMLBM_SRC_LINK;
  const Par<T> q = par_of<T>(D);
  for (int i = threadIdx.x; i < G::FZ; i += G::NT) sCol[i] = ghost_col(k0 - 3 + i, Nz, zw);
  if (threadIdx.x < G::SR) sRow[threadIdx.x] = row_of(q, j0 - 1 + (int)threadIdx.x, D.k64[K_R0]);
  __syncthreads();
  pdl_wait();
  if (MODE != 3 && gridDim.x <= G::kEarly) pdl_trigger();
  if (ctr && blockIdx.x == 0 && threadIdx.x == 0) ctr[2 + (parity ^ 1)] = ctr[2 + parity] + 1;

  // u on the tile + 3.  Ghost columns at the z walls: u odd.  Ghost rows (depth 2):
  // u_z even, u_r odd about the axis; about the outer wall u_r odd, u_z even
  // (free-slip) or odd (no-slip); beyond an inlet or outlet row b the linear
  // continuation 2 u(b) - u.
  if (ax) {
    for_sites<G::NT, G::FR, G::FZ>([&](int lr, int lc) {
      const int j = j0 - 3 + lr;
      if (j < -2 || j > Nr + 1) return;
      const int c = sCol[lc];
      T uz, ur;
      if (j >= 0 && j < Nr) {
        const int o = j * P + c;
        uz = T{uv[o]};
        ur = T{uv[plane + o]};
      } else {
        int m, b = -1;
        if (j < 0) {
          if (inl) { b = 0; m = -j; } else { m = -1 - j; }
        } else {
          if (outl) { b = Nr - 1; m = 2 * (Nr - 1) - j; } else { m = 2 * Nr - 1 - j; }
        }
        const int o = m * P + c;
        uz = T{uv[o]};
        ur = -T{uv[plane + o]};
        if (b >= 0) {
          uz = fma(lit<T>(2.0), T{uv[b * P + c]}, -uz);
          ur = fma(lit<T>(2.0), T{uv[plane + b * P + c]}, ur);
        } else if (j >= Nr && noslip) {
          uz = -uz;
        }
      }
      const int k = k0 - 3 + lc;
      if (zw && (k < 0 || k >= Nz)) {
        uz = -uz;
        ur = -ur;
      }
      sUz[lr * G::FZ + lc] = uz;
      sUr[lr * G::FZ + lc] = ur;
    });
    __syncthreads();
  }

  // Sources on the tile + 1 (half of them for the link average); an inlet or outlet
  // row has none and leaves the equilibrium of its imposed state.
  for_sites<G::NT, G::SR, G::SZ>([&](int lr, int lc) {
    const int j = j0 - 1 + lr, k = k0 - 1 + lc, si = lr * G::SZ + lc;
    if (j < 0 || j >= Nr) return;
    const bool bin = inl && j == 0, bout = outl && j == Nr - 1;
    T S_ = lit<T>(0.0), Hz = lit<T>(0.0), Hr = lit<T>(0.0);
    const int c = sCol[lc + 2];
    if (bin || bout) {
      T rho, uz, ur;
      if (bin) {
        rho = T{uv[2 * plane + P + c]};
        uz = T{D.inlet[c]};
        ur = T{D.inlet[Nz + c]};
      } else {
        const int o = (Nr - 2) * P + c;
        rho = T{D.k64[K_RHOOUT]};
        uz = T{uv[o]};
        ur = T{uv[plane + o]};
      }
      T fe[9];
      equilibrium(rho, uz, ur, fe);
#pragma unroll
      for (int i = 0; i < 9; ++i) sB[bout][i][lc] = fe[i];
    } else if (ax) {
      const int fi = (lr + 2) * G::FZ + (lc + 2);
      const T rho{uv[2 * plane + j * P + c]};
      const T druz = d1(sUz + fi, G::FZ), dzur = d1(sUr + fi, 1), drur = d1(sUr + fi, G::FZ);
      if constexpr (MODE == 3) {
        if (lr >= 1 && lr <= BR && lc >= 1 && lc <= BZ && k < Nz) {
          double* w = inter + (size_t)j * P + k;
          w[I_G1 * iplane] = unscale(druz, 12.0).v;
          w[I_G2 * iplane] = unscale(dzur, 12.0).v;
          w[I_G3 * iplane] = unscale(drur, 12.0).v;
        }
      }
      site_sources(q, rho, sUz[fi], sUr[fi], druz, dzur, drur, sRow[lr], S_, Hz, Hr);
      if (link) {
        S_ = S_ * lit<T>(0.5);
        Hz = Hz * lit<T>(0.5);
        Hr = Hr * lit<T>(0.5);
      }
    }
    if constexpr (MODE == 3) {
      if (!ax && lr >= 1 && lr <= BR && lc >= 1 && lc <= BZ && k < Nz)
        for (int g = I_G1; g <= I_G3; ++g) inter[g * iplane + (size_t)j * P + k] = 0.0;
    }
    sS[si] = S_;
    sHz[si] = Hz;
    sHr[si] = Hr;
  });

  // Streaming: every role pulls its directions; away from the boundaries direction i
  // comes from x - c_i.
  double* __restrict__ fout = static_cast<double*>(D.f[parity ^ 1]);
  double* __restrict__ psout = static_cast<double*>(D.psi[parity ^ 1]);
  const int role = ROLES > 1 ? (int)threadIdx.x / G::SITES : 0;
  bool synced = false;
  for (int t = (int)threadIdx.x - role * G::SITES; t < G::SITES; t += (ROLES > 1 ? G::SITES : G::NT)) {
    const int lr = t / BZ, lc = t - lr * BZ, j = j0 + lr, k = k0 + lc;
    const bool in = j < Nr && k < Nz;
    const bool brow = (inl && j == 0) || (outl && j == Nr - 1);
    const bool edge = j == 0 || j == Nr - 1 || (inl && j == 1) || (outl && j == Nr - 2) ||
                      (zw && (k == 0 || k == Nz - 1));
    const int km = k == 0 ? Nz - 1 : k - 1, kp = k == Nz - 1 ? 0 : k + 1;  // periodic neighbours
    const int o = j * P + k;
    T fn[9];
    if (in && !edge) {  // the loads first: they overlap the end of the sources stage
      with_role<ROLES>(role, [&](auto R) {
#pragma unroll
        for (int i = 0; i < 9; ++i)
          if (pull_role(i, ROLES) == R.value)
            fn[i] = T{fs[i * plane + (j - cr_(i)) * P + (cz_(i) == 0 ? k : cz_(i) > 0 ? km : kp)]};
      });
    }
    if (!synced) __syncthreads();  // the sources
    synced = true;
    if (in) {
      with_role<ROLES>(role, [&](auto R) {
        if (!edge) {
          if (ax) {
#pragma unroll
            for (int i = 0; i < 9; ++i) {
              if (pull_role(i, ROLES) != R.value) continue;
              const int si = (lr + 1 - cr_(i)) * G::SZ + (lc + 1 - cz_(i));
              fn[i] = add_source(i, fn[i], sS[si], sHz[si], sHr[si]);
            }
          }
        } else {
#pragma unroll
          for (int i = 0; i < 9; ++i) {
            if (pull_role(i, ROLES) != R.value) continue;
            // where the population arriving in direction i leaves from: row sj, column sk,
            // direction ii, which is i with the flagged components reversed
            int sj = j - cr_(i), sk = cz_(i) == 0 ? k : cz_(i) > 0 ? km : kp, ii = i;
            bool own = false, flip_z = false, flip_r = false;
            if (brow) {  // inlet / outlet row: its own boundary populations
              own = true;
            } else if (zw && (k - cz_(i) < 0 || k - cz_(i) >= Nz)) {  // through a z wall: bounce-back
              own = flip_z = flip_r = true; ii = opp_(i);
            } else if (sj < 0) {  // through the axis: specular reflection
              sj = j; ii = mirror_(i); flip_r = true;
            } else if (sj >= Nr) {  // through the outer wall
              sj = j; flip_r = true;
              if (noslip) { own = flip_z = true; ii = opp_(i); }
              else { ii = mirror_(i); }
            }
            int sc = lc + 1 - cz_(i);
            if (own) { sj = j; sk = k; sc = lc + 1; }
            if ((inl && sj == 0) || (outl && sj == Nr - 1)) {
              fn[i] = sB[sj != 0][ii][sc];
            } else {
              fn[i] = T{fs[ii * plane + sj * P + sk]};
              if (ax) {
                const int si = (sj - j0 + 1) * G::SZ + sc;
                const T Z = sHz[si], Rr = sHr[si];
                fn[i] = add_source(i, fn[i], sS[si], flip_z ? -Z : Z, flip_r ? -Rr : Rr);
              }
            }
          }
        }
        if (link && ax && !brow) {  // the other half, at the arrival site
          const int di = (lr + 1) * G::SZ + (lc + 1);
#pragma unroll
          for (int i = 0; i < 9; ++i)
            if (pull_role(i, ROLES) == R.value) fn[i] = add_source(i, fn[i], sS[di], sHz[di], sHr[di]);
        }
#pragma unroll
        for (int i = 0; i < 9; ++i) {
          if (pull_role(i, ROLES) != R.value) continue;
          fout[i * plane + o] = fn[i].v;
        }
        if constexpr (ROLES > 1) {
          if (R.value == 0) sF[t] = fn[0] + (fn[2] + fn[4]);
          if (R.value == 1 % ROLES) sF[G::SITES + t] = fn[1] + fn[3];
          if (R.value == 2 % ROLES) sF[2 * G::SITES + t] = fn[5] + fn[6];
          if (R.value == 3 % ROLES) sF[3 * G::SITES + t] = fn[7] + fn[8];
        }
      });
    }
    if constexpr (ROLES > 1) __syncthreads();
    if (in && role == 0) {
      T rho;
      if constexpr (ROLES > 1) rho = sF[t] + (sF[G::SITES + t] + (sF[2 * G::SITES + t] + sF[3 * G::SITES + t]));
      else rho = moment0(fn);
      psout[o] = psi_of(q, rho).v;
    }
  }
}

struct Tile64 { int tz, tr; };
constexpr Tile64 kTiles64[] = {{32, 8}, {64, 8}, {32, 16}, {16, 8}, {8, 4}};

template <int BZ, int BR>
cudaError_t step64_t(const InstDesc* d, const int* ti, int nt, int parity, cudaStream_t s, int* ctr) {
  constexpr int NT = Geo64<BZ, BR>::NT;
  const cudaError_t e = launch_pdl(f64_force<BZ, BR, 0>, nt, NT, 0, s, d, ti, 0, parity, (double*)nullptr,
                                   (size_t)0, (double*)nullptr);
  if (e != cudaSuccess) return e;
  return launch_pdl(f64_stream<BZ, BR, 0>, nt, NT, 0, s, d, ti, parity, (double*)nullptr, (size_t)0,
                    (const double*)nullptr, ctr);
}

template <int BZ, int BR>
cudaError_t readback64_t(const InstDesc* d, const int* ti, int nt, int toff, int parity, cudaStream_t s) {
  return launch_pdl(f64_force<BZ, BR, 1>, nt, Geo64<BZ, BR>::NT, 0, s, d, ti, toff, parity, (double*)nullptr,
                    (size_t)0, (double*)nullptr);
}

template <int BZ, int BR>
cudaError_t readback64_load_t() {
  cudaFuncAttributes a;
  return cudaFuncGetAttributes(&a, f64_force<BZ, BR, 1>);
}

template <int BZ, int BR>
cudaError_t inter64_t(const InstDesc* d, const int* ti, int nt, double* inter, size_t iplane, double* fstar,
                      cudaStream_t s) {
  constexpr int NT = Geo64<BZ, BR>::NT;
  const cudaError_t e = launch_pdl(f64_force<BZ, BR, 3>, nt, NT, 0, s, d, ti, 0, 0, inter, iplane, fstar);
  if (e != cudaSuccess) return e;
  return launch_pdl(f64_stream<BZ, BR, 3>, nt, NT, 0, s, d, ti, 0, inter, iplane, (const double*)fstar,
                    (int*)nullptr);
}

}  // namespace

int split64_tile_list(int* tz, int* tr, int cap) {
  int n = 0;
  for (const auto& e : kTiles64) {
    if (n < cap && tz && tr) { tz[n] = e.tz; tr[n] = e.tr; }
    ++n;
  }
  return n;
}

bool split64_tile_supported(int tz, int tr) {
  for (const auto& e : kTiles64)
    if (e.tz == tz && e.tr == tr) return true;
  return false;
}

// fn<BZ, BR>() of the tile
#define AMLBM_TILE64(fn, ...)                                      \
  if (tz == 32 && tr == 8) return fn<32, 8>(__VA_ARGS__);          \
  if (tz == 64 && tr == 8) return fn<64, 8>(__VA_ARGS__);          \
  if (tz == 32 && tr == 16) return fn<32, 16>(__VA_ARGS__);        \
  if (tz == 16 && tr == 8) return fn<16, 8>(__VA_ARGS__);          \
  if (tz == 8 && tr == 4) return fn<8, 4>(__VA_ARGS__);            \
  return cudaErrorInvalidValue;

cudaError_t launch_step_split64(int tz, int tr, const InstDesc* d, const int* ti, int nt, int parity, cudaStream_t s,
                                int* ctr) {
  if (nt <= 0) return cudaSuccess;
  AMLBM_TILE64(step64_t, d, ti, nt, parity, s, ctr)
}

cudaError_t launch_readback64(int tz, int tr, const InstDesc* d, const int* ti, int nt, int toff, int parity,
                              cudaStream_t s) {
  if (nt <= 0) return cudaSuccess;
  AMLBM_TILE64(readback64_t, d, ti, nt, toff, parity, s)
}

cudaError_t readback64_preload(int tz, int tr) {
  AMLBM_TILE64(readback64_load_t)
}

cudaError_t launch_step_inter64(int tz, int tr, const InstDesc* d, const int* ti, int nt, double* inter,
                                size_t iplane, double* fstar, cudaStream_t s) {
  if (tz == 32 && tr == 8) return inter64_t<32, 8>(d, ti, nt, inter, iplane, fstar, s);
  if (tz == 8 && tr == 4) return inter64_t<8, 4>(d, ti, nt, inter, iplane, fstar, s);
  return cudaErrorInvalidValue;
}

}  // namespace amlbm
