// Quotients by a rounded reciprocal and a correction (lbm_device.cuh) against
// the GPU's correctly rounded divisions, bit by bit: FP32, FP64, and the
// double-FP32 quotient with each of its two divisions done as a division.
// Numerators over 2^-60 .. 1, denominators 1/2 .. 2 (densities) and near 1.
#include <cstdio>
#include <cstdlib>

#include "lbm_device.cuh"

using namespace lbm::dev;

__device__ uint32_t word(uint32_t i, uint32_t k) { return fmix32(fmix32(i) ^ (0x9E3779B9u * k)); }

__global__ void check(uint32_t n, unsigned long long *bad) {
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    const uint32_t a = word(i, 1), b = word(i, 2), c = word(i, 3), d = word(i, 4);
    const float mant = __uint_as_float(0x3F800000u | (b & 0x7FFFFFu));  // [1, 2)
    const float r = i % 4 == 0 ? 1.0f + (static_cast<int>(b % 2000001u) - 1000000) * 1e-8f
                               : ((b >> 23) & 1u ? mant : 0.5f * mant);
    const float v = __uint_as_float((a & 0x807FFFFFu) | ((127u - (a >> 23) % 60u) << 23));
    if (quotient(v, r, __frcp_rn(r)) != __fdiv_rn(v, r)) atomicAdd(&bad[0], 1ull);

    const double rd = r + c * 0x1p-56, vd = v + v * (d * 0x1p-56);
    if (quotient(vd, rd, 1.0 / rd) != vd / rd) atomicAdd(&bad[1], 1ull);

    // low parts: up to half a unit in the last place of the high ones
    const DF x = df_quick(v, v * (static_cast<int>(c) * 0x1p-56f));
    const DF y = df_quick(r, r * (static_cast<int>(d) * 0x1p-56f));
    const DF got = df_div_inv(x, y, __frcp_rn(y.h));
    const float q1 = __fdiv_rn(x.h, y.h);
    const DF rem = df_sub(x, df_mul_f(y, q1));
    const DF want = df_quick(q1, __fdiv_rn(rem.h, y.h));
    if (got.h != want.h || got.l != want.l) atomicAdd(&bad[2], 1ull);
  }
}

int main() {
  unsigned long long *bad, out[3];
  const uint32_t n = 1u << 24;
  if (cudaMalloc(&bad, sizeof(out)) != cudaSuccess || cudaMemset(bad, 0, sizeof(out)) != cudaSuccess)
    return 2;
  check<<<1024, 256>>>(n, bad);
  if (cudaMemcpy(out, bad, sizeof(out), cudaMemcpyDeviceToHost) != cudaSuccess) return 2;
  std::printf("%u quotients; unlike the division: FP32 %llu, FP64 %llu, double-FP32 %llu\n", n, out[0],
              out[1], out[2]);
  return out[0] || out[1] || out[2];
}
