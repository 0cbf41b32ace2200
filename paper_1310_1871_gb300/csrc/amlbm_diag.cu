// Diagnostics of a lattice state: FP64 sums over the meridional sites and the
// interface radius of every column, for one instance or for every instance of
// a batch in the same three launches.
//
// Quantities (r = j + 1/2 + r_off is the node radius, sums over real sites):
//   mass2d = sum rho, mass3d = sum 2 pi r rho (the volume integral of the
//   axisymmetric density, Sec. II.A), momz3d = sum 2 pi r rho u_z,
//   E_ke = pi sum r rho |u|^2 (the kinetic energy whose constancy marks the
//   steady pipe flow, Sec. III.A), max |u|, the l = 2 moment a_2 of the liquid
//   fraction about the drop centre (Sec. III.C), the r-intercept of the
//   interface on the centre column and its minimum over z (the neck of a thread,
//   Sec. III.D), and the Shan-Chen pressure p = rho/3 + G psi^2/6 (the equation
//   of state of Sec. II.B with c_s^2 = 1/3) inside and outside the drop.
//
// The read-back kernel must have written rho, u_z, u_r of the state into the
// instance's rho_out / uz_out / ur_out arrays first (in the compute type C).

#include <cuda_runtime.h>

#include "amlbm.h"
#include "amlbm_internal.cuh"
#include "amlbm_launch.cuh"

namespace amlbm {
namespace {

constexpr int DIAG_NT = 256;
constexpr int DIAG_WARPS = DIAG_NT / 32;
constexpr int NSUM = 8;  // mass2d mass3d momz3d Eke q2 sumS bad | max |u|^2 (max-reduced)

// Sums v[q] over the warp, all seven at once: each of the first three exchanges also halves
// the quantities a lane still holds, so that lane l ends with the sum of quantity
// (l >> 2) & 7, bits reversed (lane_sum).  9 additions instead of 35, and one value per lane
// left to convert: FP64 operations and conversions take 64 clocks a warp.
template <class C>
__device__ __forceinline__ C warp_sums(const C* v) {
  const int lane = threadIdx.x & 31;
  C a[4], b[2];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const C hi = i < 3 ? v[4 + i] : C(0);
    a[i] = (lane & 16 ? hi : v[i]) + __shfl_xor_sync(0xffffffffu, lane & 16 ? v[i] : hi, 16);
  }
#pragma unroll
  for (int i = 0; i < 2; ++i)
    b[i] = (lane & 8 ? a[2 + i] : a[i]) + __shfl_xor_sync(0xffffffffu, lane & 8 ? a[i] : a[2 + i], 8);
  C c = (lane & 4 ? b[1] : b[0]) + __shfl_xor_sync(0xffffffffu, lane & 4 ? b[0] : b[1], 4);
  c += __shfl_xor_sync(0xffffffffu, c, 2);
  return c + __shfl_xor_sync(0xffffffffu, c, 1);
}
__device__ __forceinline__ int lane_sum(int lane) { return (lane >> 4 & 1) * 4 + (lane >> 3 & 1) * 2 + (lane >> 2 & 1); }

// Maximum and minimum of values that are never negative: their bit patterns order as
// they do, which keeps the comparison off the FP64 pipe; a NaN loses in the minimum.
__device__ __forceinline__ float warp_max_t(float v) {
  return __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(v)));
}
__device__ __forceinline__ double warp_max_t(double v) {
  unsigned long long x = __double_as_longlong(v);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) x = max(x, __shfl_xor_sync(0xffffffffu, x, o));
  return __longlong_as_double(x);
}
__device__ __forceinline__ unsigned long long bits_min(unsigned long long x) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) x = min(x, __shfl_xor_sync(0xffffffffu, x, o));
  return x;
}

// Interface radius of column k, one warp: the first row (from row 0) whose
// density is below mid, interpolated linearly against the row before it; r0 - 1/2
// (the axis, or the lattice's inner edge) when row 0 is already below, Nr + r0 - 1/2
// when no row is.  r0 is the radius of row 0.  Rows are scanned 32 at a time, the loads of
// four such groups in flight together.
template <class C>
__device__ double col_radius_warp(const C* rho, int Nz, int Nr, int k, double mid, double r0) {
  const C midc = C(mid);
  const int lane = threadIdx.x & 31;
  for (int j4 = 0; j4 < Nr; j4 += 128) {
    C v4[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int j = j4 + 32 * i + lane;
      v4[i] = j < Nr ? rho[(size_t)j * Nz + k] : midc;
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int j0 = j4 + 32 * i;
      const unsigned m = __ballot_sync(0xffffffffu, v4[i] < midc);
      if (m) {  // one lane interpolates (an FP64 division), the others take its value
        const int jf = j0 + __ffs(m) - 1;
        double res = r0 - 0.5;
        if (lane == 0 && jf > 0) {  // the fraction in C (an FP64 division is slow here)
          const C v0 = rho[(size_t)(jf - 1) * Nz + k], v = rho[(size_t)jf * Nz + k];
          res = (jf - 1 + r0) + double((v0 - midc) / (v0 - v));
        }
        return __shfl_sync(0xffffffffu, res, 0);
      }
    }
  }
  return Nr + r0 - 0.5;
}

__device__ __forceinline__ float rcp_t(float x) { return __frcp_rn(x); }
__device__ __forceinline__ double rcp_t(double x) { return __drcp_rn(x); }

// Block blk of the nblk blocks of job J: partial sums over the sites
// blk*NT + tid + m*nblk*NT into partials[(J.blk0 + blk) * NSUM + q], and the
// radii of the columns blk*WARPS + warp + m*nblk*WARPS into cols[J.col0 + k].
// The per-site terms are formed in the arithmetic type C of the storage form
// (its values are no more precise than that) and summed per thread and per warp
// in C, then across warps and blocks in FP64; FP64 runs at a small fraction of
// the FP32 rate on GB300, so there is no FP64 operation, division or square root
// per site or lane (|u|^2 is max-reduced, its root taken once at the end).  The
// FP64 form (C = double) is FP64 throughout.  Alone on a cold cache, us with four
// dependent site loads and 40 additions a warp / now: FP64 64 x 32 18.4 / 8.3, 32 x 111
// 15.7 / 7.6, FP32 256 x 128 8.0 / 5.6, the 450-row threads 43 / 29.
template <class C>
__device__ void partial_block(const InstDesc& D, const DiagJob& J, int blk, double* partials,
                              double* cols) {
  const int Nz = D.Nz, Nr = D.Nr, N = Nz * Nr;
  const C two_pi = C(2.0 * 3.14159265358979323846);
  const C inv_dl = C(J.inv_dl), rho_v = C(J.rho_v), zc = C(J.zc);
  const C r0 = sizeof(C) == 8 ? C(D.k64[K_R0]) : C(D.k32[K_R0]);
  const C* rho_o = static_cast<const C*>(D.rho_out);
  const C* uz_o = static_cast<const C*>(D.uz_out);
  const C* ur_o = static_cast<const C*>(D.ur_out);
  // Each thread first adds its own sites (one to four on lattices of at most 1,048,576
  // sites, ceil(Nz Nr / 262,144) beyond: 128 on 8192 x 4096) in C, then the block
  // and the final pass reduce those per-thread sums in FP64: the FP32 forms then
  // need one FP64 conversion and addition per sum and thread, not per site.
  C tacc[NSUM] = {C(0), C(0), C(0), C(0), C(0), C(0), C(0), C(0)};
  // sites n = blk * NT + tid + m * S, S = nblk * NT; (j, k) advanced without a
  // division per site
  const int S = J.nblk * DIAG_NT, sj = S / Nz, sk = S - sj * Nz;
  const int n0 = blk * DIAG_NT + threadIdx.x;
  int j = n0 / Nz, k = n0 - (n0 / Nz) * Nz;
  for (int n4 = n0; n4 < N; n4 += 4 * S) {  // the loads of four sites in flight together
    C rho4[4], uz4[4], ur4[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int n = n4 + i * S;  // S <= 2^18 (diag_blocks), N <= 2^30
      if (n < N) {
        rho4[i] = rho_o[n];
        uz4[i] = uz_o[n];
        ur4[i] = ur_o[n];
      }
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      if (n4 + i * S >= N) break;
      const C r = C(j) + r0, rho = rho4[i], uz = uz4[i], ur = ur4[i];
      const C u2 = uz * uz + ur * ur, w = two_pi * r * rho;
      tacc[0] += rho;
      tacc[1] += w;
      tacc[2] += w * uz;
      tacc[3] += C(0.5) * w * u2;
      const C dz = C(k) - zc;
      tacc[4] += two_pi * r * ((rho - rho_v) * inv_dl) * (dz * dz - C(0.5) * r * r);
      tacc[5] += -rho * ur * rcp_t(r);
      const bool bad = !(rho > C(0)) || !isfinite(rho) || !isfinite(u2);
      tacc[6] += bad ? C(1) : C(0);
      tacc[7] = fmax(tacc[7], bad ? C(0) : u2);
      k += sk;
      j += sj;
      if (k >= Nz) {
        k -= Nz;
        ++j;
      }
    }
  }
  // The warp's 32 sums pairwise in C too, then FP64 across warps and blocks.
  const double sum = double(warp_sums(tacc));
  const C top = warp_max_t(tacc[NSUM - 1]);
  __shared__ double red[DIAG_WARPS][NSUM];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if ((lane & 3) == 0) red[warp][lane_sum(lane)] = lane == 28 ? double(top) : sum;
  __syncthreads();
  if (threadIdx.x < NSUM) {
    const int q = threadIdx.x;
    double v = red[0][q];
#pragma unroll
    for (int w = 1; w < DIAG_WARPS; ++w) v = q == NSUM - 1 ? fmax(v, red[w][q]) : v + red[w][q];
    partials[(size_t)(J.blk0 + blk) * NSUM + q] = v;
  }
  const double mid = 0.5 * (J.rho_l + J.rho_v);
  for (int k = blk * DIAG_WARPS + warp; k < Nz; k += J.nblk * DIAG_WARPS) {
    const double rad = col_radius_warp<C>(rho_o, Nz, Nr, k, mid, D.k64[K_R0]);
    if (lane == 0) cols[J.col0 + k] = rad;
  }
}

// One block: the job's partial sums and column radii reduced into out[16].  Thread
// q + 8 s (q < 8) folds quantity q of the blocks b = s (mod 32) in FP64, shuffles and one
// pass through shared memory join them, and other warps meanwhile form the pressures and
// the radii: GB300's FP64 operations are slow, so the pass is bound by the length of its
// chains.  Alone on a cold cache, us on the 450-row threads (443 blocks a lattice) / 64 drops:
// one warp 42 / 11.4, eight warps 13.5 / 8.1.
constexpr int FINAL_NT = 256;

template <class C>
__device__ void final_block(const InstDesc& D, const DiagJob& J, int parity, const double* partials,
                            const double* cols, double* out) {
  const int Nz = D.Nz, Nr = D.Nr;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, q = lane & (NSUM - 1);
  __shared__ double red[FINAL_NT / 32][NSUM];
  __shared__ unsigned long long neck[FINAL_NT / 32];
  unsigned long long cmin = __double_as_longlong(1e300);
  for (int k = threadIdx.x; k < Nz; k += FINAL_NT)
    cmin = min(cmin, (unsigned long long)__double_as_longlong(cols[J.col0 + k]));
  double acc = 0.0;
  for (int b = threadIdx.x / NSUM; b < J.nblk; b += FINAL_NT / NSUM) {
    const double v = partials[(size_t)(J.blk0 + b) * NSUM + q];
    acc = q == NSUM - 1 ? fmax(acc, v) : acc + v;
  }
#pragma unroll
  for (int o = 8; o < 32; o <<= 1) {
    const double v = __shfl_xor_sync(0xffffffffu, acc, o);
    acc = q == NSUM - 1 ? fmax(acc, v) : acc + v;
  }
  cmin = bits_min(cmin);
  if (lane < NSUM) red[warp][lane] = acc;
  if (lane == 0) neck[warp] = cmin;
  if (warp == 1 || warp == 2) {
    int kc = (int)llround(J.zc);
    kc %= Nz;
    if (kc < 0) kc += Nz;
    if (warp == 2) {
      if (lane == 0) out[6] = cols[J.col0 + kc];
    } else {  // lane 0: the pressure inside, on the axis at the drop's centre; lane 1: outside
      const double G = D.G;
      const int k = lane == 0 ? kc : (kc + Nz / 2) % Nz, j = lane == 0 ? 0 : Nr - 1;
      double p = 0.0;
      if (lane < 2) {
        const double rho = double(static_cast<const C*>(D.rho_out)[(size_t)j * Nz + k]);
        const double ps = double(static_cast<const C*>(D.psi[parity])[(size_t)j * D.P + k]);
        p = rho / 3.0 + G * ps * ps / 6.0;
        out[8 + lane] = p;
      }
      const double po = __shfl_sync(0xffffffffu, p, 1);
      if (lane == 0) out[10] = p - po;
    }
  }
  __syncthreads();
  if (warp == 0 && lane < NSUM) {
    double t = red[0][lane];
#pragma unroll
    for (int w = 1; w < FINAL_NT / 32; ++w) t = lane == NSUM - 1 ? fmax(t, red[w][lane]) : t + red[w][lane];
    if (lane < 4) out[lane] = t;
    else if (lane == 4) out[5] = t * J.a2norm;
    else if (lane == 5) out[12] = t;
    else if (lane == 6) out[11] = t;
    else out[4] = sqrt(t);
  }
  if (warp == 3 && lane == 0) {
    unsigned long long c = neck[0];
#pragma unroll
    for (int w = 1; w < FINAL_NT / 32; ++w) c = min(c, neck[w]);
    out[7] = __longlong_as_double(c);
    out[13] = out[14] = out[15] = 0.0;
  }
}

template <class C>
__global__ void __launch_bounds__(DIAG_NT) diag_partial_one(const InstDesc* __restrict__ descs, DiagJob J,
                                                            double* partials, double* cols) {
  pdl_wait();
  pdl_trigger();
  partial_block<C>(descs[J.inst], J, blockIdx.x, partials, cols);
}

template <class C>
__global__ void __launch_bounds__(FINAL_NT) diag_final_one(const InstDesc* __restrict__ descs, DiagJob J,
                                                           int parity, const double* partials,
                                                           const double* cols, double* out) {
  pdl_wait();
  final_block<C>(descs[J.inst], J, parity, partials, cols, out);
}

// Every job of a batch: block b belongs to job blkjob[b] (the host's table of
// the jobs' block ranges [blk0, blk0 + nblk)).
template <class C>
__global__ void __launch_bounds__(DIAG_NT) diag_partial_all(const InstDesc* __restrict__ descs,
                                                            const DiagJob* __restrict__ jobs,
                                                            const int* __restrict__ blkjob,
                                                            double* partials, double* cols) {
  pdl_wait();
  pdl_trigger();
  const DiagJob J = jobs[blkjob[blockIdx.x]];
  partial_block<C>(descs[J.inst], J, blockIdx.x - J.blk0, partials, cols);
}

template <class C>
__global__ void __launch_bounds__(FINAL_NT) diag_final_all(const InstDesc* __restrict__ descs,
                                                           const DiagJob* __restrict__ jobs, int parity,
                                                           const double* partials, const double* cols,
                                                           double* out) {
  pdl_wait();
  const DiagJob J = jobs[blockIdx.x];
  final_block<C>(descs[J.inst], J, parity, partials, cols, out + (size_t)16 * blockIdx.x);
}

}  // namespace

double a2_norm(double R) { return 5.0 / (4.0 * 3.14159265358979323846 * std::pow(R, 5.0)); }

void diag_job_constants(DiagJob& J) {
  J.a2norm = a2_norm(J.R);
  J.inv_dl = 1.0 / (J.rho_l - J.rho_v);
}

// One site per thread while the pass (`sites` over all its lattices) has at most eight
// blocks per SM, then two, then four; more only where 1024 blocks a lattice (1,048,576
// sites) are not enough for that.  A batch counts the sites of all its lattices for a pass
// over one of them too, so that both passes add in the same order.
int diag_blocks(int Nz, int Nr, long long sites) {
  const long long round = 8LL * 152 * DIAG_NT;
  const int N = Nz * Nr, each = DIAG_NT * (sites <= round ? 1 : sites <= 2 * round ? 2 : 4);
  int nb = (N + each - 1) / each;
  const int nbz = (Nz + DIAG_NT - 1) / DIAG_NT;
  if (nb < nbz) nb = nbz;
  if (nb > 1024) nb = 1024;
  return nb < 1 ? 1 : nb;
}

cudaError_t launch_diag(int storage, const InstDesc* d, int inst, int Nz, int Nr, int parity,
                        double zc, double R, double rho_l, double rho_v, double* partials,
                        int nblk, double* cols, double* out, cudaStream_t s) {
  (void)Nz;
  (void)Nr;
  DiagJob J;
  J.zc = zc;
  J.R = R;
  J.rho_l = rho_l;
  J.rho_v = rho_v;
  diag_job_constants(J);
  J.inst = inst;
  J.blk0 = 0;
  J.nblk = nblk;
  J.col0 = 0;
  cudaError_t e;
  if (storage == AMLBM_STORE_F64) {
    e = launch_pdl(diag_partial_one<double>, nblk, DIAG_NT, 0, s, d, J, partials, cols);
    if (e == cudaSuccess) e = launch_pdl(diag_final_one<double>, 1, FINAL_NT, 0, s, d, J, parity, partials, cols, out);
  } else {
    e = launch_pdl(diag_partial_one<float>, nblk, DIAG_NT, 0, s, d, J, partials, cols);
    if (e == cudaSuccess) e = launch_pdl(diag_final_one<float>, 1, FINAL_NT, 0, s, d, J, parity, partials, cols, out);
  }
  return e;
}

cudaError_t diag_preload() {
  cudaFuncAttributes a;
  cudaError_t e = cudaFuncGetAttributes(&a, diag_partial_one<double>);
  if (e == cudaSuccess) e = cudaFuncGetAttributes(&a, diag_final_one<double>);
  if (e == cudaSuccess) e = cudaFuncGetAttributes(&a, diag_partial_one<float>);
  if (e == cudaSuccess) e = cudaFuncGetAttributes(&a, diag_final_one<float>);
  return e;
}

cudaError_t launch_diag_all(int storage, const InstDesc* d, const DiagJob* d_jobs, const int* d_blkjob,
                            int njobs, int total_blocks, int parity, double* partials, double* cols,
                            double* out, cudaStream_t s) {
  if (njobs < 1 || total_blocks < 1) return cudaErrorInvalidValue;
  cudaError_t e;
  if (storage == AMLBM_STORE_F64) {
    e = launch_pdl(diag_partial_all<double>, total_blocks, DIAG_NT, 0, s, d, d_jobs, d_blkjob, partials, cols);
    if (e == cudaSuccess) e = launch_pdl(diag_final_all<double>, njobs, FINAL_NT, 0, s, d, d_jobs, parity, partials, cols, out);
  } else {
    e = launch_pdl(diag_partial_all<float>, total_blocks, DIAG_NT, 0, s, d, d_jobs, d_blkjob, partials, cols);
    if (e == cudaSuccess) e = launch_pdl(diag_final_all<float>, njobs, FINAL_NT, 0, s, d, d_jobs, parity, partials, cols, out);
  }
  return e;
}

}  // namespace amlbm
