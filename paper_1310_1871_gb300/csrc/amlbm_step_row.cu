// The FP32-arithmetic timestep of small lattices on sm_103a: the chain of
// amlbm_step.cu with one warp per row and one site per thread.
//
// What bounds a step of a small lattice is neither bandwidth nor arithmetic but the
// chain of one site: few tiles, so every stage that a warp has to walk more than once
// adds its whole latency.  Here a CTA of H + 6 warps holds H x 26 sites and a halo of
// three, so that each row of the halo'd tile is 32 columns, one warp: a thread keeps its
// site's populations, collided populations and sources in registers from the first
// load to the last, and only psi, d_r psi, u and the collided populations pass
// through shared memory, with one barrier each.  Ghost rows and columns of u have no
// pass of their own: their threads compute the mirrored site over again and turn the
// signs.  The next step may start as soon as this one has begun to read (pdl_trigger): its
// blocks then wait beside this one's, with the index arithmetic and 1 / r done, since both
// fit on an SM.  us per step with the trigger at the end of the kernel / here: 64 x 32 3.65 /
// 3.24, 256 x 128 5.0 / 4.1, 512 x 128 6.1 / 5.2; the persistent kernel takes 9.9, 9.5 and
// 10.3, the strips 7.2, 7.7 and 7.7.  The arithmetic is amlbm_step.cu's, operation for
// operation: the same bits.  64 registers a thread: two CTAs of 16 warps per SM.
#include "amlbm_packed.cuh"
#include "amlbm_launch.cuh"

namespace amlbm {
namespace {

enum { M_STEP = 0, M_READ = 1, M_INTER = 3 };

// Sites of u around the tile; psi has 4 more, d_r psi 2 more.
template <int MODE> constexpr int kHalo = MODE == M_READ ? 0 : 3;
constexpr int kPz = 40, kDz = 36, kSz = 28;  // columns of psi, of d_r psi, of the collided populations
constexpr int kReadRows = 8;

template <int MODE>
__host__ __device__ constexpr int warps_of(int H) { return H + 2 * kHalo<MODE>; }
template <int MODE>
constexpr size_t smem_of(int H) {
  const int W = warps_of<MODE>(H);
  return 4 * (size_t)((W + 8) * kPz + (W + 4) * kDz + (MODE == M_READ ? 0 : 3 * W * 32 + 9 * (H + 2) * kSz));
}

// M_STEP: the timestep; M_READ: rho and u of the tile; M_INTER: the timestep and the forward
// intermediates of the state it starts from (I_COUNT planes of `iplane` elements).
template <class S, int MODE>
__global__ void __launch_bounds__(MODE == M_READ ? 32 * kReadRows : 32 * (kRowMaxRows + 6), MODE == M_READ ? 4 : 2)
    row_kernel(const InstDesc* __restrict__ descs, const int* __restrict__ tile_inst, int toff, int H, int parity,
               int* __restrict__ ctr, float* __restrict__ inter, size_t iplane) {
  using T = F1;
  constexpr int HF = kHalo<MODE>, BZ = 32 - 2 * HF, HP = HF + 4, HD = HF + 2;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, W = warps_of<MODE>(H);
  T* sPsi = reinterpret_cast<T*>(smem_raw);
  T* sDr = sPsi + (W + 8) * kPz;
  T* sUz = sDr + (W + 4) * kDz;
  T* sUr = sUz + W * 32;
  T* sRho = sUr + W * 32;  // inlet and outlet lattices only
  T* sF = sRho + W * 32;
  const int nS = (H + 2) * kSz;

  const int tile = blockIdx.x + toff;
  const InstDesc& D = descs[tile_inst[tile]];
  const int Nz = D.Nz, Nr = D.Nr, P = D.P;
  const int tz = MODE == M_READ ? D.rb_tiles_z : D.tiles_z;
  const int l = tile - (MODE == M_READ ? D.rb_tile_base : D.tile_base);
  const int k0 = (l % tz) * BZ, j0 = (l / tz) * H;
  const size_t plane = (size_t)P * Nr;
  const bool ax = D.axisym != 0, guo = D.forcing == AMLBM_FORCE_GUO, link = D.src == AMLBM_SRC_LINK;
  const bool zw = D.zbc == AMLBM_Z_NOSLIP, noslip = D.wall == AMLBM_WALL_NOSLIP;
  const bool inl = D.rlo == AMLBM_RLO_INLET, outl = D.wall == AMLBM_WALL_OUTLET;
  const int shift = D.shift;
  const Par<T> q = par_of<T>(D);
  const float rho0 = D.k32[K_RHO0], rref = D.k32[K_RREF], inv_rho0 = D.k32[K_INVRHO0];

  // This thread's slot (j, k) and the site (js, at lane ls) it computes: beyond a
  // reflecting wall the mirrored one, whose u it takes with the wall's signs.
  const int j = j0 - HF + w, k = k0 - HF + lane;
  int js = j, ls = lane;
  bool odd_z = false, odd_r = false;
  if constexpr (HF > 0) {
    if (j < 0 && !inl) {
      js = -1 - j;
      odd_r = true;
    } else if (j >= Nr && !outl) {
      js = 2 * Nr - 1 - j;
      odd_r = true;
      odd_z = noslip;
    }
    if (zw && (k == -1 || k == -2 || k == Nz || k == Nz + 1)) {
      ls = lane + (k < 0 ? -1 - 2 * k : 2 * (Nz - k) - 1);
      odd_z = !odd_z;
      odd_r = !odd_r;
    }
  }
  const bool on = js >= 0 && js < Nr && j >= -2 && j < Nr + 2;
  const int lr = js - (j0 - HF);
  const Row<T> row = {T{rcp_one(__fadd_rn(__int2float_rn(js), D.k32[K_R0]))}};
  const size_t at = (size_t)(on ? js : 0) * P + ghost_col(k, Nz, zw);
  const size_t pr0 = (size_t)ghost_row(j0 - HP + w, Nr, inl, outl) * P;
  const size_t pr1 = (size_t)ghost_row(j0 - HP + w + W, Nr, inl, outl) * P;
  const int pc0 = ghost_col(k0 - HP + lane, Nz, zw), pc1 = ghost_col(k0 - HP + 32 + lane, Nz, zw);
  const S* fin = static_cast<const S*>(D.f[parity]) + at;
  const float* psin = static_cast<const float*>(D.psi[parity]);

  pdl_wait();
  pdl_trigger();
  uint32_t step = 0;
  if constexpr (MODE == M_STEP) {  // the step's number, for the stochastic rounding
    if (sizeof(S) == 2 || (tile == 0 && threadIdx.x == 0)) step = (uint32_t)ctr[2 + parity];
    if (tile == 0 && threadIdx.x == 0) ctr[2 + (parity ^ 1)] = (int)(step + 1);
  }

  // psi of the tile + 4 beyond the slots, and the site's populations
  const bool second = w < 8, extra = lane < kPz - 32;
  const float a0 = __ldcg(psin + pr0 + pc0), a1 = extra ? __ldcg(psin + pr0 + pc1) : 0.0f;
  const float b0 = second ? __ldcg(psin + pr1 + pc0) : 0.0f, b1 = second && extra ? __ldcg(psin + pr1 + pc1) : 0.0f;
  S fq[9];
  float vz = 0.0f, vr = 0.0f;
  if (on) {
#pragma unroll
    for (int i = 0; i < 9; ++i) fq[i] = __ldcg(fin + i * plane);
    if (shift == 3) {
      vz = __ldcg(psin + at + plane);
      vr = __ldcg(psin + at + 2 * plane);
    }
  }
  sPsi[w * kPz + lane] = T{a0};
  if (extra) sPsi[w * kPz + 32 + lane] = T{a1};
  if (second) {
    sPsi[(w + W) * kPz + lane] = T{b0};
    if (extra) sPsi[(w + W) * kPz + 32 + lane] = T{b1};
  }
  __syncthreads();

  // isotropic d_r psi, 2 beyond the slots
  if (ax) {
    const T* p = sPsi + (w + HP - HD) * kPz + lane + HP - HD;
    T* o = sDr + w * kDz + lane;
    const bool more = lane < kDz - 32;
    o[0] = iso_r(p, kPz);
    if (more) o[32] = iso_r(p + 32, kPz);
    if (w < 4) {
      o[W * kDz] = iso_r(p + W * kPz, kPz);
      if (more) o[W * kDz + 32] = iso_r(p + W * kPz + 32, kPz);
    }
    __syncthreads();
  }

  // moments, forces, u; the collided populations stay in fs
  T fs[9], rho = lit<T>(0.0), uz = rho, ur = rho;
  if (on) {
    const T* p = sPsi + (lr + HP - HF) * kPz + ls + HP - HF;
    const T psi = p[0];
    T f[9];
    decode_values<S>(shift, fq, psi.v, vz, vr, inv_rho0, rho0, rref, f);
    rho = moment0(f);
    const T jz = moment_z(f), jr = moment_r(f);
    T sz, sr, dr0 = lit<T>(0.0), Drr = dr0, Dzr = dr0;
    sc_sums(p, kPz, sz, sr);
    if (ax) {
      const T* dr = sDr + (lr + HD - HF) * kDz + ls + HD - HF;
      dr0 = dr[0];
      Drr = iso_r(dr, kDz);
      T e[5];
#pragma unroll
      for (int m = -2; m <= 2; ++m) e[m + 2] = m ? d1(p + m, kPz) : lit<T>(0.0);
      Dzr = d1(e + 2, 1);
    }
    T Fz, Fr;
    forces(q, rho, psi, sz, sr, ax, dr0, Drr, Dzr, row, Fz, Fr);
    const T inv_rho = {rcp_one(rho.v)};
    uz = fma(Fz, lit<T>(0.5), jz) * inv_rho;
    ur = fma(Fr, lit<T>(0.5), jr) * inv_rho;
    if constexpr (MODE == M_READ) {
      if (k < Nz) {
        const size_t o = (size_t)j * Nz + k;
        static_cast<float*>(D.rho_out)[o] = rho.v;
        static_cast<float*>(D.uz_out)[o] = uz.v;
        static_cast<float*>(D.ur_out)[o] = ur.v;
      }
    } else {
      const T tz_ = odd_z ? -uz : uz, tr_ = odd_r ? -ur : ur;
      sUz[w * 32 + lane] = tz_;
      sUr[w * 32 + lane] = tr_;
      if (inl || outl) sRho[w * 32 + lane] = rho;
      collide(q, guo, T{D.k32[K_GUO]}, f, rho, uz, ur, jz, jr, Fz, Fr, inv_rho, [&](int i, T v) { fs[i] = v; });
      if constexpr (MODE == M_INTER) {
        if (w >= HF && w < HF + H && lane >= HF && lane < HF + BZ && j < Nr && k < Nz) {
          float* o = inter + (size_t)j * P + k;
          o[I_RHO * iplane] = rho.v;
          o[I_UZ * iplane] = uz.v;
          o[I_UR * iplane] = ur.v;
          o[I_VZ * iplane] = (fma(Fz, q.tau, jz) * inv_rho).v;
          o[I_VR * iplane] = (fma(Fr, q.tau, jr) * inv_rho).v;
          o[I_FZ * iplane] = Fz.v;
          o[I_FR * iplane] = Fr.v;
          o[I_PSI * iplane] = psi.v;
          o[I_SZ * iplane] = sz.v;
          o[I_SR * iplane] = sr.v;
          o[I_DR * iplane] = dr0.v;
          o[I_DRR * iplane] = Drr.v;
          o[I_DZR * iplane] = Dzr.v;
        }
      }
    }
  }
  if constexpr (MODE != M_READ) {
    __syncthreads();

    // Beyond an inlet or outlet row b: u(b - m) = 2 u(b) - u(b + m).
    if (ax && ((inl && j0 < HF) || (outl && j0 + H + HF > Nr))) {
      const bool lo = inl && (j == -1 || j == -2), hi = outl && (j == Nr || j == Nr + 1);
      if (lo || hi) {
        const int b = lo ? 0 : Nr - 1, m = 2 * b - j;
        const int bi = (b - (j0 - HF)) * 32 + lane, mi = (m - (j0 - HF)) * 32 + lane;
        sUz[w * 32 + lane] = fma(lit<T>(2.0), sUz[bi], -sUz[mi]);
        sUr[w * 32 + lane] = fma(lit<T>(2.0), sUr[bi], -sUr[mi]);
      }
      __syncthreads();
    }

    // velocity gradients and sources of the tile + 1; the populations that leave its sites
    T h[9];
    const bool brow = (inl && j == 0) || (outl && j == Nr - 1);
    if (w >= HF - 1 && w <= HF + H && lane >= HF - 1 && lane <= HF + BZ && j >= 0 && j < Nr) {
      const int fi = w * 32 + lane;
      if (brow) {
        // the equilibrium of the imposed velocity and row 1's density (inlet), of the
        // imposed density and row Nr - 2's velocity (outlet); no source
        const int nb = fi + (j == 0 && inl ? 32 : -32);
        if (inl && j == 0) {
          const int kk = ghost_col(k, Nz, zw);
          equilibrium(sRho[nb], T{(float)D.inlet[kk]}, T{(float)D.inlet[Nz + kk]}, fs);
        } else {
          equilibrium(T{D.k32[K_RHOOUT]}, sUz[nb], sUr[nb], fs);
        }
      } else if (ax) {
        const T druz = d1(sUz + fi, 32), dzur = d1(sUr + fi, 1), drur = d1(sUr + fi, 32);
        if constexpr (MODE == M_INTER) {
          if (w >= HF && w < HF + H && lane >= HF && lane < HF + BZ && k < Nz) {
            float* o = inter + (size_t)j * P + k;
            o[I_G1 * iplane] = druz.v;
            o[I_G2 * iplane] = dzur.v;
            o[I_G3 * iplane] = drur.v;
          }
        }
        T S_, Hz, Hr;
        site_sources(q, rho, odd_z ? -uz : uz, odd_r ? -ur : ur, druz, dzur, drur, row, S_, Hz, Hr);
        sources(S_, Hz, Hr, h);
        if (link) {
#pragma unroll
          for (int i = 0; i < 9; ++i) fs[i] = fma(h[i], lit<T>(0.5), fs[i]);
        } else {
#pragma unroll
          for (int i = 0; i < 9; ++i) fs[i] = fs[i] + h[i];
        }
      }
      if constexpr (MODE == M_INTER) {
        if (!ax && w >= HF && w < HF + H && lane >= HF && lane < HF + BZ && k < Nz) {
          float* o = inter + (size_t)j * P + k;
          o[I_G1 * iplane] = 0.0f;
          o[I_G2 * iplane] = 0.0f;
          o[I_G3 * iplane] = 0.0f;
        }
      }
      T* o = sF + (w - HF + 1) * kSz + lane - HF + 1;
#pragma unroll
      for (int i = 0; i < 9; ++i) o[i * nS] = fs[i];
    }
    __syncthreads();

    // Pull streaming of the tile (boundary maps as in amlbm_step.cu), psi, store.
    if (w >= HF && w < HF + H && lane >= HF && lane < HF + BZ && j < Nr && k < Nz) {
      const T* o = sF + (w - HF + 1) * kSz + lane - HF + 1;
      T fn[9];
      if (!(j == 0 || j == Nr - 1 || (zw && (k == 0 || k == Nz - 1)))) {
#pragma unroll
        for (int i = 0; i < 9; ++i) fn[i] = o[i * nS - cr_(i) * kSz - cz_(i)];
      } else {
#pragma unroll
        for (int i = 0; i < 9; ++i) {
          int dr = cr_(i) * kSz, dz = cz_(i), ii = i;
          const int kf = k - cz_(i);
          if (brow) {
            dr = 0; dz = 0;
          } else if (zw && (kf < 0 || kf >= Nz)) {
            dr = 0; dz = 0; ii = opp_(i);
          } else if (cr_(i) > 0 && j == 0) {
            dr = 0; ii = mirror_(i);
          } else if (cr_(i) < 0 && j == Nr - 1) {
            dr = 0;
            if (noslip) { dz = 0; ii = opp_(i); }
            else { ii = mirror_(i); }
          }
          fn[i] = o[ii * nS - dr - dz];
        }
      }
      if (link && !brow) {
        if (ax) {
#pragma unroll
          for (int i = 0; i < 9; ++i) fn[i] = fma(h[i], lit<T>(0.5), fn[i]);
        } else {  // as amlbm_step.cu, which adds its zero sources
#pragma unroll
          for (int i = 0; i < 9; ++i) fn[i] = fn[i] + lit<T>(0.0);
        }
      }
      const T rn = moment0(fn);
      const size_t so = (size_t)j * P + k;
      encode_site<S>(shift, static_cast<S*>(D.f[parity ^ 1]) + so, static_cast<float*>(D.psi[parity ^ 1]) + so, plane,
                     fn, rn, psi_of(q, rn).v, inv_rho0, rho0, rref, D.rounding, (uint32_t)(j * Nz + k), step);
    }
  }
}

template <class S>
cudaError_t step_t(const InstDesc* d, const int* ti, int nt, int H, int parity, cudaStream_t s, int* ctr) {
  static_assert(smem_of<M_STEP>(kRowMaxRows) <= 48 * 1024, "within the default shared-memory limit");
  return launch_pdl(row_kernel<S, M_STEP>, nt, 32 * warps_of<M_STEP>(H), smem_of<M_STEP>(H), s, d, ti, 0, H, parity,
                    ctr, nullptr, 0);
}
template <class S>
cudaError_t read_t(const InstDesc* d, const int* ti, int nt, int toff, int parity, cudaStream_t s) {
  return launch_pdl(row_kernel<S, M_READ>, nt, 32 * kReadRows, smem_of<M_READ>(kReadRows), s, d, ti, toff, kReadRows,
                    parity, nullptr, nullptr, 0);
}

}  // namespace

cudaError_t launch_step_row(int storage, int H, const InstDesc* d, const int* ti, int nt, int parity, cudaStream_t s,
                            int* ctr) {
  if (nt <= 0) return cudaSuccess;
  if (!ctr || !row_rows_ok(H)) return cudaErrorInvalidValue;
  switch (storage) {
    case AMLBM_STORE_F32: return step_t<float>(d, ti, nt, H, parity, s, ctr);
    case AMLBM_STORE_F16: return step_t<__half>(d, ti, nt, H, parity, s, ctr);
    case AMLBM_STORE_BF16: return step_t<__nv_bfloat16>(d, ti, nt, H, parity, s, ctr);
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t launch_readback_row(int storage, const InstDesc* d, const int* ti, int nt, int toff, int parity,
                                cudaStream_t s) {
  if (nt <= 0) return cudaSuccess;
  switch (storage) {
    case AMLBM_STORE_F32: return read_t<float>(d, ti, nt, toff, parity, s);
    case AMLBM_STORE_F16: return read_t<__half>(d, ti, nt, toff, parity, s);
    case AMLBM_STORE_BF16: return read_t<__nv_bfloat16>(d, ti, nt, toff, parity, s);
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t readback_row_preload(int storage) {
  cudaFuncAttributes a;
  switch (storage) {
    case AMLBM_STORE_F32: return cudaFuncGetAttributes(&a, row_kernel<float, M_READ>);
    case AMLBM_STORE_F16: return cudaFuncGetAttributes(&a, row_kernel<__half, M_READ>);
    case AMLBM_STORE_BF16: return cudaFuncGetAttributes(&a, row_kernel<__nv_bfloat16, M_READ>);
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t launch_step_inter_row(int H, const InstDesc* d, const int* ti, int nt, float* inter, size_t iplane,
                                  cudaStream_t s) {
  if (nt <= 0) return cudaSuccess;
  if (!row_rows_ok(H)) return cudaErrorInvalidValue;
  return launch_pdl(row_kernel<float, M_INTER>, nt, 32 * warps_of<M_INTER>(H), smem_of<M_INTER>(H), s, d, ti, 0, H, 0,
                    nullptr, inter, iplane);
}

}  // namespace amlbm
