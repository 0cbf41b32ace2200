// Checks of amlbm_packed.cuh: the packed operations round as the scalar ones do, also
// where a product feeds a sum (no contraction), and the reciprocal equals __frcp_rn for
// every 32-bit argument.  Prints "ok" or the number of differences of each check.
#include <cstdio>

#include "amlbm_packed.cuh"

using namespace amlbm;

static __device__ float number(uint32_t x) {  // a value of either sign between 2^-8 and 2^8
  const uint32_t h = mix32(x);
  return __uint_as_float((h & 0x807fffffu) | ((119u + mix32(x * 3 + 5) % 16) << 23));
}

__global__ void operations(unsigned* bad) {
  const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
  const float a = number(6 * i), b = number(6 * i + 1), c = number(6 * i + 2);
  const float d = number(6 * i + 3), e = number(6 * i + 4), f = number(6 * i + 5);
  const F2 A = pack(a, d), B = pack(b, e), C = pack(c, f);
  auto check = [&](int k, F2 got, float x, float y) {
    if (lo(got) != x || hi(got) != y) atomicAdd(bad + k, 1u);
  };
  check(0, A + B, __fadd_rn(a, b), __fadd_rn(d, e));
  check(1, A - B, __fsub_rn(a, b), __fsub_rn(d, e));
  check(2, A * B, __fmul_rn(a, b), __fmul_rn(d, e));
  check(3, fma(A, B, C), __fmaf_rn(a, b, c), __fmaf_rn(d, e, f));
  check(4, fma(A, B, C) * B + A, __fadd_rn(__fmul_rn(__fmaf_rn(a, b, c), b), a),
        __fadd_rn(__fmul_rn(__fmaf_rn(d, e, f), e), d));
  check(5, C - (A - B) * B, __fsub_rn(c, __fmul_rn(__fsub_rn(a, b), b)), __fsub_rn(f, __fmul_rn(__fsub_rn(d, e), e)));
  check(6, rcp(A), __frcp_rn(a), __frcp_rn(d));
}

__global__ void reciprocals(unsigned* bad) {
  const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x, n = gridDim.x * blockDim.x;
  for (uint64_t x = i; x < (1ull << 32); x += n) {
    const float v = __uint_as_float((uint32_t)x), got = rcp_one(v), want = __frcp_rn(v);
    if (__float_as_uint(got) != __float_as_uint(want) && !(got != got && want != want)) atomicAdd(bad + 7, 1u);
  }
}

int main() {
  unsigned *bad, host[8];
  if (cudaMalloc(&bad, sizeof(host)) != cudaSuccess || cudaMemset(bad, 0, sizeof(host)) != cudaSuccess) return 2;
  operations<<<4096, 256>>>(bad);
  reciprocals<<<4096, 256>>>(bad);
  if (cudaMemcpy(host, bad, sizeof(host), cudaMemcpyDeviceToHost) != cudaSuccess) return 2;
  bool ok = true;
  for (int k = 0; k < 8; ++k)
    if (host[k]) {
      printf("check %d: %u differences\n", k, host[k]);
      ok = false;
    }
  if (ok) printf("ok\n");
  return ok ? 0 : 1;
}
