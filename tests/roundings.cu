// Counts for test_gpu_roundings.py: how often the library's own roots and quotients differ
// from the correctly rounded ones.
#include <cstdint>

#include <cuda_runtime.h>

#include "internal.cuh"
#include "philox.cuh"
#include "reflector.cuh"

// out[0]: words x whose rho_root(-2 ln u) is not the correctly rounded root, u as in box_muller4.
__global__ void rho_kernel(unsigned long long* out) {
  unsigned n = 0;
  for (uint64_t x = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; x >> 32 == 0; x += (uint64_t)gridDim.x * blockDim.x) {
    const float u = __fmaf_rn(__uint2float_rn((uint32_t)x), 0x1p-32f, 0x1p-33f);
    const float v = __fmul_rn(-2.0f, logf(u));
    n += __float_as_uint(tts::rho_root(v)) != __float_as_uint(__fsqrt_rn(v));
  }
  if (n) atomicAdd(out, (unsigned long long)n);
}

// Norms g and heads x0 = f sqrt(g), |f| < 1, from Philox words: out[1], out[2] roots and
// quotients that are not the nearest, out[3], out[4] the largest distance in units of the last place.
__global__ void reflector_kernel(unsigned long long* out, uint64_t total) {
  unsigned nr = 0, nq = 0;
  unsigned long long dr = 0, dq = 0;
  for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < total; i += (uint64_t)gridDim.x * blockDim.x) {
    uint32_t a = (uint32_t)i, b = (uint32_t)(i >> 32), c = 7, d = 9;
    tts::philox4x32_10(a, b, c, d, 1u, 2u);
    const int e = 41 + (int)(c % 1958u);
    const double g = __hiloint2double((e << 20) | (int)(a >> 12), (int)b);
    const double f = ((double)d - 2147483648.0) * 0x1p-31, x0 = f * sqrt(g);
    double alpha, be, v0;
    tts::reflector(g, x0, alpha, be, v0);
    const double s = __dsqrt_rn(g), q = __ddiv_rn(1.0, fma(fabs(x0), fabs(alpha), g));
    const unsigned long long er = llabs(__double_as_longlong(fabs(alpha)) - __double_as_longlong(s));
    const unsigned long long eq = llabs(__double_as_longlong(be) - __double_as_longlong(q));
    nr += er != 0;
    nq += eq != 0;
    dr = er > dr ? er : dr;
    dq = eq > dq ? eq : dq;
  }
  if (nr) atomicAdd(out + 1, (unsigned long long)nr);
  if (nq) atomicAdd(out + 2, (unsigned long long)nq);
  atomicMax(out + 3, dr);
  atomicMax(out + 4, dq);
}

extern "C" int count_roundings(unsigned long long* out_dev, unsigned long long total) {
  rho_kernel<<<2048, 256>>>(out_dev);
  reflector_kernel<<<2048, 256>>>(out_dev, total);
  return (int)cudaDeviceSynchronize();
}
