// Strip kernel of the pair schedule for sm_103a (arXiv:1310.1871, Sec. II): one warp
// marches along r over a strip of the lattice, two adjacent z-sites per lane.
//
// A tile kernel passes each tile through barrier-separated stages in shared memory:
// halo work in both directions (the force region of a 64 x 24 tile is 1.41 times its
// sites, its psi region 1.98 times), every stencil tap a shared-memory load, and half
// of the issue slots lost to barriers.  Here a warp holds 64 columns and keeps the
// stencils' rows in registers while it moves up in r, so each row is computed once:
//
//   psi row r  -> isotropic and 1D d_r psi of row r - 2 (Sec. II.D), Shan-Chen sums of
//   row r - 1 (Eq. scforce) -> d_rr psi, d_zr psi, the force, moments, u, u^eq and the
//   BGK collision of row r - 4 -> velocity gradients and sources (Eq. condition_h) of
//   row r - 6 -> streaming, psi and store of row r - 7
//
// Neighbours in z come by warp shuffles, and no warp waits for another.  All arithmetic
// is on packed pairs (amlbm_packed.cuh), one issue slot for both sites.  A strip is 48
// columns (64 less 8 on either side: the chain reaches 7 sites) and H rows, with 14
// rows of which only the first stages are needed at its lower end (about 3.5 rows'
// work).  A lattice of at most 64 columns is one strip without a halo: its lanes wrap
// around the period.
//
// What bounds it: the FMA pipe's operand bandwidth, with the two warps of a sub-partition
// that 220 registers a thread allow.  A row is 224 packed operations; one with three distinct
// operand pairs takes 3.2 clocks of its SM sub-partition, any other 2.2 (measured on loops of
// them), together about 580 of the 710 clocks a row takes.  Counters of a step of 8192 x 1024
// (ncu): FMA pipe 53 % and issue slots 48 % active, DRAM 59 %; per issued instruction a warp
// waits 0.9 cycles at fixed latencies, 0.4 for shared memory and shuffles, 0.4 unselected.
// Three warps at 168 registers, with the delayed
// values in shared memory, were slower (8192 x 4096: 714 against 592 us).
// Measured (GB300, FP32 storage, us per step; the 64 x 24 tile kernel before): the 64-drop
// sweep of 835,240 sites 37.7 -> 21.5, eight threads of 3.6 M sites 119.7 -> 64.1,
// 8192 x 4096 995 -> 521 (80 B per site: 76 % of the measured HBM bandwidth),
// 256 x 128 9.5 (fused 32 x 8) -> 7.6, 255 x 65 10.3 (fused) -> 8.1.
// Read-back (the chain up to the velocity, 12 warps per SM): 8192 x 4096 diagnostics 675 ->
// 538 us, the sweep's 57 -> 48 (pair tiles of 64 x 16 before).
//
// The operations on a site's values are those of the other schedules, in their order, so
// the states are bit-identical.

#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include <stdint.h>

#include <type_traits>

#include "amlbm.h"
#include "amlbm_internal.cuh"
#include "amlbm_launch.cuh"
#include "amlbm_packed.cuh"
#include "amlbm_vec2.cuh"

namespace amlbm {
namespace {

constexpr int kRingBytes = 4 * 9 * 32 * 8;  // collided populations of four rows
constexpr unsigned kAll = 0xffffffffu;

// A row's pairs as the stencils read them: the pair, and the pairs one and two sites to
// the left and to the right of it.
struct Row5 {
  F2 c, l1, r1, l2, r2;
};
__device__ __forceinline__ Row5 neighbours(F2 c, int left, int right) {
  float a, b;
  unpack(c, a, b);
  const float la = __shfl_sync(kAll, a, left), lb = __shfl_sync(kAll, b, left);
  const float ra = __shfl_sync(kAll, a, right), rb = __shfl_sync(kAll, b, right);
  return {c, pack(lb, a), pack(b, ra), pack(la, lb), pack(ra, rb)};
}
// The pair whose values come from one site to the left / right.
__device__ __forceinline__ F2 from_left(F2 c, int left) {
  float a, b;
  unpack(c, a, b);
  return pack(__shfl_sync(kAll, b, left), a);
}
__device__ __forceinline__ F2 from_right(F2 c, int right) {
  float a, b;
  unpack(c, a, b);
  return pack(b, __shfl_sync(kAll, a, right));
}
// Minus link8 (amlbm_physics.cuh) of the row `one` and the row `two` beyond it.
__device__ __forceinline__ F2 link_n(F2 one, F2 two) { return fma(lit<F2>(-8.0), one, two); }
// d1 from its four taps
__device__ __forceinline__ F2 diff1(F2 p1, F2 m1, F2 p2, F2 m2) {
  return fma(lit<F2>(8.0), p1 - m1, m2 - p2) * lit<F2>(1.0 / 12.0);
}

// Rows in flight: a lane's pairs of psi, of the nine populations and, for the
// equilibrium shift, of the velocity, copied asynchronously into shared memory four
// rows ahead (a warp has one or two others to hide a load behind, so the distance has
// to, and registers for it would cost a third of the warps).  A lane reads only what it
// copied itself, so its own wait is enough.  Every access is a volatile asm: they keep
// their order, and a slot is read before the copy that refills it is issued.
template <class S>
struct Flight {
  static constexpr int kPair = 2 * sizeof(S);                       // bytes of a pair of populations
  static constexpr int kPops = 0, kPsi = 9 * 32 * kPair, kVel = kPsi + 32 * 8, kSlot = kVel + 2 * 32 * 8;
  static constexpr int kBytes = 4 * kSlot;                          // four slots, one per phase
};
template <int BYTES>
__device__ __forceinline__ void copy_in(uint32_t dst, const void* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"(dst), "l"(src), "n"(BYTES));
}
__device__ __forceinline__ void commit_copies() { asm volatile("cp.async.commit_group;"); }
__device__ __forceinline__ void wait_copies_but_3() { asm volatile("cp.async.wait_group 3;"); }
__device__ __forceinline__ F2 take8(uint32_t src) {
  F2 r;
  asm volatile("ld.shared.b64 %0, [%1];" : "=l"(r.v) : "r"(src));
  return r;
}
template <class S>
__device__ __forceinline__ F2 take_pair(uint32_t src) {  // a pair of populations, widened
  if constexpr (sizeof(S) == 4) {
    return take8(src);
  } else {
    uint32_t x;
    asm volatile("ld.shared.b32 %0, [%1];" : "=r"(x) : "r"(src));
    if constexpr (std::is_same<S, __half>::value) {  // Store<__half>::to, its scale on the pair
      const float2 v = __half22float2(*reinterpret_cast<const __half2*>(&x));
      return pack(v.x, v.y) * lit<F2>(1.0 / 1024.0);
    } else {
      return pack(__uint_as_float(x << 16), __uint_as_float(x & 0xffff0000u));
    }
  }
}
// A pair of a row: at columns k and k + 1, or with ODD one site at a time, at k and k2 (a
// lattice of odd width has pairs across its seam, and rows that start off the pairs).
template <bool ODD, class S>
__device__ __forceinline__ void copy_pair(uint32_t dst, const S* __restrict__ row, int k, int k2) {
  if constexpr (ODD) {
    static_assert(sizeof(S) == 4, "asynchronous copies are at least four bytes");
    copy_in<4>(dst, row + k);
    copy_in<4>(dst + 4, row + k2);
  } else {
    copy_in<2 * (int)sizeof(S)>(dst, row + k);
  }
}
template <class S, bool ODD>
__device__ __forceinline__ void copy_pops(uint32_t slot, const S* __restrict__ f, const float* __restrict__ psi,
                                          int plane, int o, int k, int k2, int shift, int lane) {
  using Q = Flight<S>;
#pragma unroll
  for (int i = 0; i < 9; ++i)
    copy_pair<ODD>(slot + Q::kPops + (i * 32 + lane) * Q::kPair, f + (size_t)i * plane + o, k, k2);
  if (shift == 3) {
    copy_pair<ODD>(slot + Q::kVel + lane * 8, psi + (size_t)plane + o, k, k2);
    copy_pair<ODD>(slot + Q::kVel + (32 + lane) * 8, psi + (size_t)2 * plane + o, k, k2);
  }
}
// The pair's values to p and p + 1; with ODD the second only if the lattice has it.
template <bool ODD, class S>
__device__ __forceinline__ void store2(S* p, S a, S b, bool second) {
  if constexpr (ODD) {
    p[0] = a;
    if (second) p[1] = b;
  } else {
    st2<S>(p, a, b);
  }
}

// decode_values on a pair, from its slot
template <class S>
__device__ __forceinline__ void decode_pair(uint32_t slot, int lane, int shift, F2 psi, float inv_rho0, float rho0,
                                            float rref, F2* f) {
  using Q = Flight<S>;
#pragma unroll
  for (int i = 0; i < 9; ++i) f[i] = take_pair<S>(slot + Q::kPops + (i * 32 + lane) * Q::kPair);
  if (shift == 0) return;
  float pa, pb;
  unpack(psi, pa, pb);
  const F2 s = pack(shift_base(shift, pa, inv_rho0, rho0, rref), shift_base(shift, pb, inv_rho0, rho0, rref));
  if (shift == 3) {
    F2 fe[9];
    equilibrium(s, take8(slot + Q::kVel + lane * 8), take8(slot + Q::kVel + (32 + lane) * 8), fe);
#pragma unroll
    for (int i = 0; i < 9; ++i) f[i] = f[i] + fe[i];
  } else {
#pragma unroll
    for (int i = 0; i < 9; ++i) f[i] = fma(lit<F2>(w_(i)), s, f[i]);
  }
}

// encode_values on a pair, and the store
template <class S, bool ODD>
__device__ __forceinline__ void store_pair(int shift, const F2* fn, F2 rho, F2 psi, float inv_rho0, float rho0,
                                           float rref, int rounding, uint32_t site, uint32_t step, S* __restrict__ f,
                                           float* __restrict__ ps, int plane, int o, bool second) {
  float pa, pb;
  unpack(psi, pa, pb);
  F2 base[9];
  if (shift == 0) {
#pragma unroll
    for (int i = 0; i < 9; ++i) base[i] = fn[i];
  } else {
    const F2 s = pack(shift_base(shift, pa, inv_rho0, rho0, rref), shift_base(shift, pb, inv_rho0, rho0, rref));
    if (shift == 3) {
      const F2 ir = rcp(rho), vz = moment_z(fn) * ir, vr = moment_r(fn) * ir;
      F2 fe[9];
      equilibrium(s, vz, vr, fe);
#pragma unroll
      for (int i = 0; i < 9; ++i) base[i] = fn[i] - fe[i];
      store2<ODD>(ps + (size_t)plane + o, lo(vz), hi(vz), second);
      store2<ODD>(ps + (size_t)2 * plane + o, lo(vr), hi(vr), second);
    } else {
#pragma unroll
      for (int i = 0; i < 9; ++i) base[i] = fma(lit<F2>(-w_(i)), s, fn[i]);
    }
  }
  uint32_t xa = 0, xb = 0;
  const bool random = sizeof(S) == 2 && rounding;
  if (random) {
    const uint32_t m = mix32(step + 0x9E3779B9u);
    xa = mix32(site ^ m);
    xb = mix32((site + 1) ^ m);
  }
#pragma unroll
  for (int i = 0; i < 9; ++i) {
    float a, b;
    S* out = f + (size_t)i * plane + o;
    if (random) {
      unpack(base[i], a, b);
      xa = lcg_next(xa);
      xb = lcg_next(xb);
      st2<S>(out, Store<S>::from_sr(a, xa), Store<S>::from_sr(b, xb));
    } else if constexpr (std::is_same<S, __half>::value) {  // Store<__half>::from, its scale on the pair
      unpack(base[i] * lit<F2>(1024.0), a, b);
      *reinterpret_cast<__half2*>(out) = __floats2half2_rn(a, b);
    } else if constexpr (std::is_same<S, __nv_bfloat16>::value) {
      unpack(base[i], a, b);
      *reinterpret_cast<__nv_bfloat162*>(out) = __floats2bfloat162_rn(a, b);
    } else {
      unpack(base[i], a, b);
      store2<ODD>(out, a, b, second);
    }
  }
  store2<ODD>(ps + o, pa, pb, second);
}

// One strip.  FORM: the shift code of a batch whose lattices are all axisymmetric with
// the velocity shift and the storage form's default rounding, so that nothing in the
// marching loop branches on the lattice's options; or kAnyForm.
// ODD: lattices of odd width among them (FP32 storage).  READ: no step, but rho and u of
// the strip's rows into the read-back planes: the chain up to the velocity, which
// reaches 4 sites, so the strip is 56 columns wide and starts 4 rows early.
constexpr int kAnyForm = -1;
template <class S, int FORM, bool ODD, bool READ>
__device__ __forceinline__ void march(const InstDesc& D, int tile, int H, int parity, int* __restrict__ ctr,
                                      F2* __restrict__ ring, uint32_t flight) {
  constexpr int kHalo = READ ? 4 : 8, kWidth = 64 - 2 * kHalo, kEarly = READ ? 4 : 7;
  static_assert(READ ? kWidth == kStripReadWidth : kWidth == kStripWidth, "the tiling of the host");
  const int lane = threadIdx.x;
  const int Nz = D.Nz, Nr = D.Nr, P = D.P, plane = P * Nr;
  const int l = tile - (READ ? D.rb_tile_base : D.tile_base), tz = READ ? D.rb_tiles_z : D.tiles_z;
  const bool whole = Nz <= 64 && (!ODD || Nz % 2 == 0);  // the strip is the whole period
  const int n = Nz >> 1;
  const int j0 = (l / tz) * H, j1 = min(j0 + H, Nr);
  const int col = whole ? 2 * lane : (l % tz) * kWidth - kHalo + 2 * lane;
  const int kk = ODD ? wrapz(col, Nz)
                     : whole ? (col < Nz ? col : 0) : (col < 0 ? col + Nz : (col >= Nz ? col - Nz : col));
  const int k2 = ODD ? wrapz(col + 1, Nz) : kk + 1;
  const int left = whole && lane == 0 ? n - 1 : (lane + 31) & 31;
  const int right = whole && lane == n - 1 ? 0 : (lane + 1) & 31;
  const bool mine = (whole || (lane >= kHalo / 2 && lane < 32 - kHalo / 2)) && col < Nz, second = col + 1 < Nz;
  const S* __restrict__ fin = static_cast<const S*>(D.f[parity]);
  const float* __restrict__ psin = static_cast<const float*>(D.psi[parity]);
  S* __restrict__ fout = static_cast<S*>(D.f[parity ^ 1]);
  float* __restrict__ psout = static_cast<float*>(D.psi[parity ^ 1]);
  constexpr bool ANY = FORM == kAnyForm;
  const bool ax = !ANY || D.axisym != 0, guo = ANY && D.forcing == AMLBM_FORCE_GUO;
  const int shift = ANY ? D.shift : FORM;
  const int rounding = ANY ? D.rounding : (std::is_same<S, __nv_bfloat16>::value && FORM == 2 ? 1 : 0);
  const bool noslip = D.wall == AMLBM_WALL_NOSLIP;
  const Par<F2> q = par_of<F2>(D);
  const F2 gk = splat<F2>(D.k32[K_GUO]);
  const float rho0 = D.k32[K_RHO0], inv_rho0 = D.k32[K_INVRHO0], rref = D.k32[K_RREF], r0 = D.k32[K_R0];
  ring += lane;  // [phase][9][32 lanes]; a lane reads only what it wrote

  // Rows kept in registers, indexed by the phase (the iteration modulo four) in which
  // they were made.
  F2 C[4];            // psi of rows r - 1 .. r - 4
  F2 L1[2], R1[2];    // its neighbours one site aside, rows r - 1 and r - 2
  F2 EZ[2] = {lit<F2>(0.0), lit<F2>(0.0)};  // the difference across, rows r - 1 and r - 2
  F2 L2, R2;          // two sites aside, row r - 1
  F2 D0[4], D1s[4];   // minus the lower links of d_r psi, made three rows ahead
  F2 SZ[4], SR[4];    // Shan-Chen sums of rows r - 1 .. r - 4
  F2 Cd[2], Ld1, Rd1, Ld2, Rd2, E0[4], E1s[4];  // the same of d_r psi (row r - 2)
  F2 X[2];            // 1D d_r psi of rows r - 3, r - 4
  F2 UZ[4], UR[4], RHO[2];  // u of rows j - 1 .. j - 4, rho of j - 1, j - 2 (j = r - 4)
  F2 MID[3], UP[3], UPP[3];  // collided populations with c_r = 0 of row s - 1, c_r = 1 of s - 1, s - 2
  float NI[2];        // -1 / radius of rows j - 1, j - 2
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    C[i] = D0[i] = D1s[i] = SZ[i] = SR[i] = E0[i] = E1s[i] = UZ[i] = UR[i] = lit<F2>(0.0);
    if (i < 2) { L1[i] = R1[i] = Cd[i] = X[i] = lit<F2>(0.0); RHO[i] = lit<F2>(1.0); NI[i] = 0.0f; }
    if (i < 3) MID[i] = UP[i] = UPP[i] = lit<F2>(0.0);
  }
  L2 = R2 = Ld1 = Rd1 = Ld2 = Rd2 = lit<F2>(0.0);

  int jb = 0;
  float nirs = 0.0f;
  using Q = Flight<S>;
  auto copy_psi = [&](int r, int ph) {
    copy_pair<ODD>(flight + ph * Q::kSlot + Q::kPsi + lane * 8, psin + reflect_row(r, Nr) * P, kk, k2);
  };
  pdl_wait();  // everything above reads only what creation wrote
  uint32_t step = 0;
  if constexpr (!READ) {
    step = (uint32_t)ctr[2 + parity];
    if (blockIdx.x == 0 && lane == 0) ctr[2 + (parity ^ 1)] = (int)(step + 1);
  }
#pragma unroll
  for (int ph = 0; ph < 4; ++ph) {
    copy_psi(j0 - kEarly + ph, ph);
    commit_copies();
  }

  // Row r of psi enters; PH is r's phase.  F_ON, S_ON: the collision row r - 4 and the
  // source row r - 6 are inside the strip's region.  F_NEXT: the collision row of four
  // rows later is.
  auto row = [&](int r, auto PHc, auto F_NEXTc, auto F_ONc, auto S_ONc) {
    constexpr int PH = decltype(PHc)::value, P1 = PH & 1;
    constexpr bool F_NEXT = decltype(F_NEXTc)::value, F_ON = decltype(F_ONc)::value, S_ON = decltype(S_ONc)::value;
    const uint32_t slot = flight + PH * Q::kSlot;
    wait_copies_but_3();
    const F2 pc = take8(slot + Q::kPsi + lane * 8);
    F2 f[9];
    if constexpr (F_ON) decode_pair<S>(slot, lane, shift, C[PH], inv_rho0, rho0, rref, f);  // row r - 4
    copy_psi(r + 4, PH);
    if constexpr (F_NEXT)
      copy_pops<S, ODD>(slot, fin, psin, plane, min(max(r, 0), Nr - 1) * P, kk, k2, shift, lane);
    commit_copies();
    const Row5 p = neighbours(pc, left, right);

    // Shan-Chen sums of row r - 1
    const F2 c1 = C[(PH + 3) & 3], c2 = C[(PH + 2) & 3], c3 = C[(PH + 1) & 3], c4 = C[PH];
    const F2 l1 = L1[P1 ^ 1], r1 = R1[P1 ^ 1], l1b = L1[P1], r1b = R1[P1];
    const F2 e = p.r1 - p.l1;
    SZ[PH] = fma(EZ[P1 ^ 1], lit<F2>(1.0 / 9.0), (e + EZ[P1]) * lit<F2>(1.0 / 36.0));
    EZ[P1] = e;
    SR[PH] = fma(p.c - c2, lit<F2>(1.0 / 9.0), ((p.r1 - r1b) + (p.l1 - l1b)) * lit<F2>(1.0 / 36.0));
    // isotropic d_r psi and 1D d_r psi of row r - 2
    const F2 dr = ((link_n(c1, p.c) - D0[(PH + 1) & 3]) +
                   ((link_n(r1, p.r2) + link_n(l1, p.l2)) - D1s[(PH + 1) & 3])) * lit<F2>(-1.0 / 36.0);
    const F2 x = diff1(c1, c3, p.c, c4);
    D0[PH] = link_n(p.c, c1);  // for row r + 1
    D1s[PH] = link_n(p.r1, R2) + link_n(p.l1, L2);
    C[PH] = p.c;
    L1[P1] = p.l1;
    R1[P1] = p.r1;
    L2 = p.l2;
    R2 = p.r2;

    const Row5 d = neighbours(dr, left, right);  // row r - 2
    const F2 drr = ((link_n(Cd[P1 ^ 1], d.c) - E0[(PH + 1) & 3]) +
                    ((link_n(Rd1, d.r2) + link_n(Ld1, d.l2)) - E1s[(PH + 1) & 3])) * lit<F2>(-1.0 / 36.0);
    const F2 dr0 = Cd[P1], x0 = X[P1];  // row r - 4
    E0[PH] = link_n(d.c, Cd[P1 ^ 1]);
    E1s[PH] = link_n(d.r1, Rd2) + link_n(d.l1, Ld2);
    Cd[P1] = d.c;
    X[P1] = x;
    Ld1 = d.l1;
    Rd1 = d.r1;
    Ld2 = d.l2;
    Rd2 = d.r2;

    if constexpr (F_ON) {
      const int j = r - 4;
      const F2 psi = c4;
      const float nir = __shfl_sync(kAll, nirs, j - jb);
      const F2 sz = SZ[(PH + 1) & 3], sr = SR[(PH + 1) & 3];
      const F2 gpsi = psi * q.negG;
      F2 Fz = gpsi * sz, Fr = gpsi * sr;
      if (ax) {
        const Row5 e = neighbours(x0, left, right);
        const F2 dzr = diff1(e.r1, e.l1, e.r2, e.l2);
        const F2 g = (psi * q.gfac) * splat<F2>(-nir);
        Fz = fma(g, dzr, Fz);
        Fr = fma(g, fma(dr0, splat<F2>(nir), drr), Fr);
      }
      const F2 rho = moment0(f), jz = moment_z(f), jr = moment_r(f);
      Fz = fma(rho, q.gz, Fz);
      const F2 inv_rho = rcp(rho);
      F2 uz = fma(Fz, lit<F2>(0.5), jz) * inv_rho, ur = fma(Fr, lit<F2>(0.5), jr) * inv_rho;
      if constexpr (READ) {
        if (mine && j < j1) {
          const int w = j * Nz + col;
          store2<ODD>(static_cast<float*>(D.rho_out) + w, lo(rho), hi(rho), second);
          store2<ODD>(static_cast<float*>(D.uz_out) + w, lo(uz), hi(uz), second);
          store2<ODD>(static_cast<float*>(D.ur_out) + w, lo(ur), hi(ur), second);
        }
        return;
      }
      collide(q, guo, gk, f, rho, uz, ur, jz, jr, Fz, Fr, inv_rho,
              [&](int i, F2 v) { ring[(PH * 9 + i) * 32] = v; });
      // Ghost rows of u (depth 2): rows -1, -2 mirror rows 0, 1 about the axis (u_z even,
      // u_r odd) as those arrive; rows Nr, Nr + 1 mirror rows Nr - 1, Nr - 2 about the
      // outer wall (u_r odd, u_z even for free-slip and odd for no-slip).
      if (j <= 1 || j >= Nr) {
        if (j == 0) { UZ[(PH + 3) & 3] = uz; UR[(PH + 3) & 3] = negate(ur); }
        if (j == 1) { UZ[(PH + 1) & 3] = uz; UR[(PH + 1) & 3] = negate(ur); }
        if (j == Nr) { uz = UZ[(PH + 3) & 3]; ur = negate(UR[(PH + 3) & 3]); }
        if (j == Nr + 1) { uz = UZ[(PH + 1) & 3]; ur = negate(UR[(PH + 1) & 3]); }
        if (j >= Nr && noslip) uz = negate(uz);
      }

      if constexpr (S_ON) {
        const int s = r - 6, o = r - 7;
        F2 g[9];
#pragma unroll
        for (int i = 0; i < 9; ++i) g[i] = ring[(((PH + 2) & 3) * 9 + i) * 32];
        if (ax) {
          const F2 us = UR[(PH + 2) & 3];
          const F2 druz = diff1(UZ[(PH + 3) & 3], UZ[(PH + 1) & 3], uz, UZ[PH]);
          const F2 drur = diff1(UR[(PH + 3) & 3], UR[(PH + 1) & 3], ur, UR[PH]);
          const Row5 e = neighbours(us, left, right);
          const F2 dzur = diff1(e.r1, e.l1, e.r2, e.l2);
          add_sources(q, RHO[P1], UZ[(PH + 2) & 3], us, druz, dzur, drur, splat<F2>(NI[P1]), g);
        }
        // arrivals in row o from row s (c_r = -1), s - 1 (c_r = 0) and s - 2 (c_r = 1)
        F2 down[3] = {g[4], from_right(g[7], right), from_left(g[8], left)};
        const F2 up[3] = {g[2], from_left(g[5], left), from_right(g[6], right)};
        if (s >= Nr - 1) {
          // through the outer wall, row Nr - 1's own populations: reversed in r at the same
          // place they left for (free-slip) or where they started (no-slip); kept for the
          // next row in the ring slot that row's collision would have
          F2* w = ring + ((PH + 3) & 3) * 9 * 32;
          if (s == Nr - 1) {
            w[0] = up[0];
            w[32] = noslip ? g[5] : up[2];
            w[64] = noslip ? g[6] : up[1];
          } else {
            w = ring + ((PH + 2) & 3) * 9 * 32;
            down[0] = w[0];
            down[1] = w[32];
            down[2] = w[64];
          }
        }
        if (o >= j0 && o < j1) {
          const F2 fn[9] = {MID[0], MID[1], UPP[0], MID[2], down[0], UPP[1], UPP[2], down[1], down[2]};
          const F2 rn = moment0(fn);
          const F2 pn = psi_of(q, rn);
          if (mine)
            store_pair<S, ODD>(shift, fn, rn, pn, inv_rho0, rho0, rref, rounding, (uint32_t)(o * Nz + col), step, fout,
                                 psout, plane, o * P + col, second);
        }
#pragma unroll
        for (int i = 0; i < 3; ++i) {
          UPP[i] = UP[i];
          UP[i] = up[i];
        }
        if (s == 0) {  // through the axis: row 0's own populations, reversed in r
          UPP[0] = down[0];
          UPP[1] = down[2];
          UPP[2] = down[1];
        }
        MID[0] = g[0];
        MID[1] = from_left(g[1], left);
        MID[2] = from_right(g[3], right);
      }
      UZ[PH] = uz;
      UR[PH] = ur;
      RHO[P1] = rho;
      NI[P1] = nir;
    }
  };
  // -1 / radius of 32 rows from jb on, one per lane
  auto radii = [&](int from) {
    jb = from;
    nirs = -rcp_one(__fadd_rn(__int2float_rn(jb + lane), r0));
  };
  using std::integral_constant;
  using Off = integral_constant<bool, false>;
  using On = integral_constant<bool, true>;
  int r = j0 - kEarly;
  auto rows4 = [&](auto F_NEXTc, auto F_ONc, auto S_ONc) {
    row(r, integral_constant<int, 0>(), F_NEXTc, F_ONc, S_ONc);
    row(r + 1, integral_constant<int, 1>(), F_NEXTc, F_ONc, S_ONc);
    row(r + 2, integral_constant<int, 2>(), F_NEXTc, F_ONc, S_ONc);
    row(r + 3, integral_constant<int, 3>(), F_NEXTc, F_ONc, S_ONc);
    r += 4;
  };
  rows4(Off(), Off(), Off());
  rows4(On(), Off(), Off());
  radii(r - 4);
  rows4(On(), On(), Off());
  using Rest = integral_constant<bool, !READ>;
#pragma unroll 1
  while (r < j1 + kEarly) {
    if (r - 4 - jb == 32) radii(r - 4);
    rows4(On(), On(), Rest());
  }
  asm volatile("cp.async.wait_all;");
}

template <class S, int FORM, bool ODD>
__global__ void __launch_bounds__(32, 8) strip_step(const InstDesc* __restrict__ descs,
                                                    const int* __restrict__ tile_inst, int H, int parity,
                                                    int* __restrict__ ctr) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  march<S, FORM, ODD, false>(descs[tile_inst[blockIdx.x]], blockIdx.x, H, parity, ctr,
                             reinterpret_cast<F2*>(smem_raw),
                             (uint32_t)__cvta_generic_to_shared(smem_raw) + kRingBytes);
  pdl_trigger();
}

template <class S, int FORM, bool ODD>
__global__ void __launch_bounds__(32, 12) strip_read(const InstDesc* __restrict__ descs,
                                                     const int* __restrict__ tile_inst, int toff, int H, int parity) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int tile = blockIdx.x + toff;
  march<S, FORM, ODD, true>(descs[tile_inst[tile]], tile, H, parity, nullptr, nullptr,
                            (uint32_t)__cvta_generic_to_shared(smem_raw));
  pdl_trigger();
}

// What to launch: a step or a read-back of nt tiles from toff, or the loading of the
// read-back's code.
struct Call {
  enum { kStep, kRead, kLoad } kind;
  int form, H, nt, toff, parity;
  bool odd;
  const InstDesc* d;
  const int* ti;
  cudaStream_t s;
  int* ctr;
};

template <class S, int FORM, bool ODD>
cudaError_t issue(const Call& c) {
  constexpr size_t smem = kRingBytes + Flight<S>::kBytes;
  static_assert(smem <= 48 * 1024, "within the default shared-memory limit");
  if (c.kind == Call::kStep)
    return launch_pdl(strip_step<S, FORM, ODD>, c.nt, 32, smem, c.s, c.d, c.ti, c.H, c.parity, c.ctr);
  // the read-back branches on the shift of the 16-bit forms
  constexpr int F = sizeof(S) == 4 ? FORM : kAnyForm;
  if (c.kind == Call::kRead)
    return launch_pdl(strip_read<S, F, ODD>, c.nt, 32, (size_t)Flight<S>::kBytes, c.s, c.d, c.ti, c.toff, c.H,
                      c.parity);
  cudaFuncAttributes a;
  return cudaFuncGetAttributes(&a, strip_read<S, F, ODD>);
}

cudaError_t choose(int storage, const Call& c) {
  if (c.odd) {
    if (storage != AMLBM_STORE_F32) return cudaErrorInvalidValue;
    return c.form == 0 ? issue<float, 0, true>(c) : issue<float, kAnyForm, true>(c);
  }
  switch (storage) {
    case AMLBM_STORE_F32: return c.form == 0 ? issue<float, 0, false>(c) : issue<float, kAnyForm, false>(c);
    case AMLBM_STORE_F16:
      return c.form == 2   ? issue<__half, 2, false>(c)
             : c.form == 3 ? issue<__half, 3, false>(c)
                           : issue<__half, kAnyForm, false>(c);
    case AMLBM_STORE_BF16:
      return c.form == 2   ? issue<__nv_bfloat16, 2, false>(c)
             : c.form == 3 ? issue<__nv_bfloat16, 3, false>(c)
                           : issue<__nv_bfloat16, kAnyForm, false>(c);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace

cudaError_t launch_step_strip(int storage, int form, bool odd, int H, const InstDesc* d, const int* ti, int nt,
                              int parity, cudaStream_t s, int* ctr) {
  if (nt <= 0) return cudaSuccess;
  if (!ctr) return cudaErrorInvalidValue;
  return choose(storage, {Call::kStep, form, H, nt, 0, parity, odd, d, ti, s, ctr});
}

cudaError_t launch_readback_strip(int storage, int form, bool odd, int H, const InstDesc* d, const int* ti, int nt,
                                  int toff, int parity, cudaStream_t s) {
  if (nt <= 0) return cudaSuccess;
  return choose(storage, {Call::kRead, form, H, nt, toff, parity, odd, d, ti, s, nullptr});
}

cudaError_t readback_strip_preload(int storage, int form, bool odd) {
  return choose(storage, {Call::kLoad, form, 0, 0, 0, 0, odd, nullptr, nullptr, nullptr, nullptr});
}

}  // namespace amlbm
