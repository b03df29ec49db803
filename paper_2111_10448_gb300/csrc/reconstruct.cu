// Reconstruction X~(i_1..i_d) = G_1(:, i_1, :) ... G_d(:, i_d, :) (Sec. 2.2)
// and its fused relative-error form (eq. (1.1)).
//
// The cores are contracted into a left interface L_{d*} (N_{d*} x r_{d*}) and a
// right interface Rt_{d*+1} (r_{d*} x M_{d*}); then X~ = L_{d*} Rt_{d*+1} seen as
// the middle unfolding: digit arithmetic on the tensor cores for larger FP32 data
// (expand.cuh), else one thread per entry (FP64).
#include <algorithm>

#include "expand.cuh"
#include "internal.cuh"

namespace tts {
namespace {

constexpr int kThreads = 256;

// L_k(u + N_{k-1} i, c) = sum_a L_{k-1}(u, a) G_k(a, i, c);  L_0 = [1].
__global__ void iface_left_kernel(const double* Lp, int64_t Np, int rpp, const double* G, int64_t nk,
                                  int rpk, double* Lo) {
  const int64_t Nk = Np * nk;
  const int64_t total = Nk * rpk;
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < total;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t row = e % Nk;
    const int c = (int)(e / Nk);
    const int64_t u = row % Np, i = row / Np;
    double acc = 0.0;
    if (Lp == nullptr) {
      acc = G[0 + rpp * (i + nk * c)];
    } else {
      for (int a = 0; a < rpp; ++a) acc += Lp[u + Np * a] * G[a + rpp * (i + nk * c)];
    }
    Lo[row + Nk * c] = acc;
  }
}

// Rt_k(a, i + n_k v) = sum_c G_k(a, i, c) Rt_{k+1}(c, v);  Rt_{d+1} = [1].
__global__ void iface_right_kernel(const double* Rn, int64_t Mn, int rpn, const double* G, int64_t nk,
                                   int rpa, double* Ro) {
  const int64_t Mk = nk * Mn;
  const int64_t total = (int64_t)rpa * Mk;
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < total;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int a = (int)(e % rpa);
    const int64_t col = e / rpa;
    const int64_t i = col % nk, v = col / nk;
    double acc = 0.0;
    if (Rn == nullptr) {
      acc = G[a + rpa * (i + nk * 0)];
    } else {
      for (int c = 0; c < rpn; ++c) acc += G[a + rpa * (i + nk * c)] * Rn[c + rpn * v];
    }
    Ro[a + (int64_t)rpa * col] = acc;
  }
}

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// X~(u + Nm v) = sum_c L(u, c) Rt(c, v); optionally store it and/or accumulate
// [sum (X - X~)^2, sum X^2].
__global__ void __launch_bounds__(kThreads) dense_kernel(const double* L, const double* Rt, int64_t Nm,
                                                         int64_t Mm, int rp, void* out, int out_f64,
                                                         const void* Xc, int xc_f64, double* out2) {
  double e2 = 0.0, x2 = 0.0;
  const int64_t total = Nm * Mm;
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < total;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t u = e % Nm, v = e / Nm;
    double acc = 0.0;
    for (int c = 0; c < rp; ++c) acc += L[u + Nm * c] * Rt[c + (int64_t)rp * v];
    if (out) {
      if (out_f64) ((double*)out)[e] = acc;
      else ((float*)out)[e] = (float)acc;
    }
    if (Xc) {
      const double x = xc_f64 ? ((const double*)Xc)[e] : (double)((const float*)Xc)[e];
      e2 += (x - acc) * (x - acc);
      x2 += x * x;
    }
  }
  if (out2) {
    __shared__ double red[2][32];
    e2 = warp_sum(e2);
    x2 = warp_sum(x2);
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if (lane == 0) {
      red[0][wid] = e2;
      red[1][wid] = x2;
    }
    __syncthreads();
    if (wid == 0) {
      double a = lane < (int)(blockDim.x >> 5) ? red[0][lane] : 0.0;
      double b = lane < (int)(blockDim.x >> 5) ? red[1][lane] : 0.0;
      a = warp_sum(a);
      b = warp_sum(b);
      if (lane == 0) {
        atomicAdd(out2, a);
        atomicAdd(out2 + 1, b);
      }
    }
  }
}

// Y(row, c) += sum_v dX(row + Nk v) Rt(c, v)   (Rt: rp x Mk, ld rp).
// A job is 32 consecutive rows (the lanes) x vc consecutive v; the four warps
// of a block take consecutive jobs of the same rows, add their partial sums in
// shared memory and the block adds them into Y (FP64 atomics).  RP >= rp is a
// compile-time bound so that the accumulators stay in registers.
template <int RP>
__global__ void __launch_bounds__(128) ygram_kernel(const void* dX, int dx_f64, int64_t Nk, int64_t Mk,
                                                    const double* Rt, int rp, double* Y, int64_t vc) {
  extern __shared__ double part[];  // 4 x RP x 32
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t nrb = (Nk + 31) / 32, nvc = (Mk + vc - 1) / vc;
  const int64_t nvg = (nvc + 3) / 4;  // groups of four v chunks, one per warp
  for (int64_t job = blockIdx.x; job < nrb * nvg; job += gridDim.x) {
    const int64_t rb = job % nrb, vg = job / nrb;
    const int64_t row = rb * 32 + lane;
    const int64_t v0 = (vg * 4 + warp) * vc, v1 = imin64(Mk, v0 + vc);
    double acc[RP];
#pragma unroll
    for (int c = 0; c < RP; ++c) acc[c] = 0.0;
    if (row < Nk) {
      for (int64_t v = v0; v < v1; ++v) {
        const int64_t idx = row + Nk * v;
        const double x = dx_f64 ? __ldg((const double*)dX + idx) : (double)__ldg((const float*)dX + idx);
#pragma unroll
        for (int c = 0; c < RP; ++c)
          if (c < rp) acc[c] += x * __ldg(Rt + c + (int64_t)rp * v);
      }
    }
    __syncthreads();
#pragma unroll
    for (int c = 0; c < RP; ++c) part[(warp * RP + c) * 32 + lane] = acc[c];
    __syncthreads();
    for (int e = threadIdx.x; e < rp * 32; e += blockDim.x) {
      const int c = e >> 5, l = e & 31;
      const int64_t r = rb * 32 + l;
      if (r < Nk) {
        const double sum = part[(0 * RP + c) * 32 + l] + part[(1 * RP + c) * 32 + l] +
                           part[(2 * RP + c) * 32 + l] + part[(3 * RP + c) * 32 + l];
        atomicAdd(Y + r + Nk * c, sum);
      }
    }
  }
}

// W(c, v) += sum_u L(u, c) dX(u + Nk v)   (L: Nk x rp; W: rp x Mk).  A warp takes V
// columns v and uc rows u, its lanes the rows: RP V sums per lane, folded over the
// lanes by a halving butterfly that leaves sum j on lane j (mod 32), one FP64
// atomic each.  Like ygram_kernel it is bound by the FP64 pipe: one FMA per entry
// and rank.
template <int RP, int V>
__global__ void __launch_bounds__(128) wgram_kernel(const void* dX, int dx_f64, int64_t Nk, int64_t Mk, const double* L,
                                                    int rp, double* W, int64_t uc) {
  constexpr int NS = RP * V;
  const int lane = threadIdx.x & 31;
  const int64_t nvg = (Mk + V - 1) / V, nuc = (Nk + uc - 1) / uc;
  const int64_t nwarps = (int64_t)gridDim.x * (blockDim.x >> 5);
  for (int64_t job = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); job < nvg * nuc; job += nwarps) {
    const int64_t v0 = (job % nvg) * V, u0 = (job / nvg) * uc, u1 = imin64(Nk, u0 + uc);
    double acc[NS];
#pragma unroll
    for (int j = 0; j < NS; ++j) acc[j] = 0.0;
    for (int64_t u = u0 + lane; u < u1; u += 32) {
      double x[V];
#pragma unroll
      for (int q = 0; q < V; ++q) {
        const int64_t e = u + Nk * imin64(v0 + q, Mk - 1);   // a column past the end is dropped below
        x[q] = dx_f64 ? __ldg((const double*)dX + e) : (double)__ldg((const float*)dX + e);
      }
#pragma unroll
      for (int c = 0; c < RP; ++c) {
        const double l = __ldg(L + u + Nk * min(c, rp - 1));
#pragma unroll
        for (int q = 0; q < V; ++q) acc[q * RP + c] = fma(l, x[q], acc[q * RP + c]);
      }
    }
#pragma unroll
    for (int b = 0; b < NS; b += 32) {
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        const bool up = lane & o;
#pragma unroll
        for (int j = 0; j < o; ++j) {
          const double keep = up ? acc[b + j + o] : acc[b + j], send = up ? acc[b + j] : acc[b + j + o];
          acc[b + j] = keep + __shfl_xor_sync(0xffffffffu, send, o);
        }
      }
      const int j = b + lane, c = j % RP;
      const int64_t v = v0 + j / RP;
      if (c < rp && v < Mk) atomicAdd(W + c + (int64_t)rp * v, acc[b]);
    }
  }
}

// The two products with dX in FP32, in digit arithmetic (digits.cuh): C(o, j) += sum_k
// x(o, k) F(k, j), o the rows u and k the columns v of dX (ROWS, F = Rt^T: Z), or the
// reverse (F = L: W).  The FP64 pipe bounds the kernels above (1.7 FMAs per cycle and
// SM); here a block takes 64 outputs and a range of the contraction, 64 at a time:
// the 64 x 64 tile of dX goes through shared memory (loaded along u either way, the
// next one in flight meanwhile), a warp scales one output's 64 values by their largest
// exponent and writes their eight digits, likewise the columns of F, and each 16 x 8
// tile of sums takes the digit products of weight up to seven of half the 64 (8 x 32
// x 2^14 < 2^24: exact in FP32), then adds them to its FP64 sums.  A value keeps 61 bits
// below the largest of its 64, and a sum of 32 products is off by at most 32 2^-57 of the two
// largest factors' product (pairs of weight eight and more); where the factors' magnitudes
// say that this is not small against sum |x F| (digit::weak), the 32 products are FP64
// FMAs.  So an entry is held to 2^-44 of sum |x F| at worst, and for random factors is
// closer than FP64 FMAs.  NB column octets.  (The digits' 16-byte chunks are swizzled by their
// row instead of padded: two CTAs an SM up to NB = 4.)
// Measured (the whole adjoint, FP64 products and these): 32^5 of rank 8 1.22 -> 0.76 ms,
// 64^4 of rank 16 1.15 -> 0.57, 48^4 of rank 40 1.30 -> 0.57, 32^4 of rank 8 120 -> 87 us (0.62, 0.47,
// 0.50 ms and 83 us with seven digits and no test of the terms; where every sum
// is formed in FP64 after all, 4000 x 4000 takes 0.80 ms at rank 6, 1.39 at 16, 3.6 at 40, FP64 throughout 0.93,
// 1.49, 3.0).
// Entries from which they serve (FP32 dX, both sides at least one tile wide): 512 x 512 of
// rank 8 72 -> 47 us, 256 x 256 74 -> 47, of rank 32 109 -> 67.
constexpr int64_t kDxMin = 1 << 16;
constexpr int kDxP = 8, kDxK = 64, kDxRaw = kDxK + 1;
__host__ __device__ constexpr int dx_smem(int nb) {
  return 2 * kDxP * (64 + 8 * nb) * kDxK + 4 * 64 * kDxRaw + 4 * (64 + 8 * nb);
}
// An FP32 value as FP64 without the conversion instruction (FP64-pipe rate).
__device__ __forceinline__ double widen(float x) {
  const uint32_t b = __float_as_uint(x), e = (b >> 23) & 255u;
  if (e - 1u >= 254u) return (double)x;   // zero, subnormal, infinite, NaN
  return __hiloint2double((int)((b & 0x80000000u) | (((b & 0x7fffffffu) >> 3) + (896u << 20))), (int)(b << 29));
}
// s + sum_k x(k) F(k) in FP64.
__device__ __noinline__ double dx_dot(const float* x, int sx, const double* F, int64_t fk, int n, double s) {
#pragma unroll 8
  for (int k = 0; k < n; ++k) s = fma((double)x[k * sx], __ldg(F + k * fk), s);
  return s;
}
template <int NB, bool ROWS>
__global__ void __launch_bounds__(256, NB <= 4 ? 2 : 1)
    dx_gemm_kernel(const float* X, int64_t Nk, int64_t Mk, const double* F, int64_t fk, int64_t fj, int rp, double* C,
                   int64_t co, int64_t cj, int64_t chunks) {
  using namespace digit;
  constexpr int P = kDxP, LEAD = 5, B = 8 * (P - 1) + LEAD, NW = P, ROWS_D = 64 + 8 * NB;
  extern __shared__ __align__(16) char dsm[];
  uint16_t* Dg = reinterpret_cast<uint16_t*>(dsm);                         // [P][ROWS_D][kDxK]
  float* raw = reinterpret_cast<float*>(dsm + 2 * P * ROWS_D * kDxK);     // [v][u], ld kDxRaw
  int* er = reinterpret_cast<int*>(raw + 64 * kDxRaw);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, gq = lane >> 2, tq = lane & 3;
  const int64_t O = ROWS ? Nk : Mk, K = ROWS ? Mk : Nk, o0 = 64 * (int64_t)blockIdx.x;
  const int64_t nch = (K + 63) / 64, c0 = (int64_t)blockIdx.y * chunks, c1 = imin64(nch, c0 + chunks);
  float nx[16];
  auto fetch = [&](int64_t ch) {
#pragma unroll
    for (int q = 0; q < 16; ++q) {
      const int e = tid + 256 * q;
      const int64_t u = (ROWS ? o0 : 64 * ch) + (e & 63), v = (ROWS ? 64 * ch : o0) + (e >> 6);
      nx[q] = u < Nk && v < Mk ? __ldg(X + u + Nk * v) : 0.0f;
    }
  };
  double c[NB][4];
#pragma unroll
  for (int q = 0; q < NB; ++q) c[q][0] = c[q][1] = c[q][2] = c[q][3] = 0.0;
  int bad = 0;
  auto put = [&](int r, double x0, double x1) {   // one digit column, two values a lane
    bad |= (undigital(x0) || undigital(x1)) ? 1 : 0;
    const int m = __reduce_max_sync(0xffffffffu, max(exp_of(x0), exp_of(x1)));
    if (lane == 0) er[r] = m;
    uint32_t d0[P], d1[P];
    digits<P>(fixed<B>(x0, m), d0);
    digits<P>(fixed<B>(x1, m), d1);
#pragma unroll
    for (int p = 0; p < P; ++p)
      *reinterpret_cast<uint32_t*>(Dg + (p * ROWS_D + r) * kDxK + 8 * ((lane >> 2) ^ (r & 7)) + 2 * (lane & 3)) =
          d0[p] | (d1[p] << 16);
  };
  if (c0 < c1) fetch(c0);
  for (int64_t ch = c0; ch < c1; ++ch) {
    __syncthreads();   // the products of the chunk before
#pragma unroll
    for (int q = 0; q < 16; ++q) {
      const int e = tid + 256 * q;
      raw[(e >> 6) * kDxRaw + (e & 63)] = nx[q];
    }
    double fx[NB][2];
#pragma unroll
    for (int q = 0; q < NB; ++q)
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        const int64_t k = 64 * ch + 2 * lane + e;
        const int j = warp + 8 * q;
        fx[q][e] = j < rp && k < K ? __ldg(F + k * fk + j * fj) : 0.0;
      }
    __syncthreads();
    if (ch + 1 < c1) fetch(ch + 1);
#pragma unroll 2
    for (int r = warp; r < 64; r += 8) {
      const float* p = ROWS ? raw + 2 * lane * kDxRaw + r : raw + r * kDxRaw + 2 * lane;
      put(r, widen(p[0]), widen(p[ROWS ? kDxRaw : 1]));
    }
#pragma unroll
    for (int q = 0; q < NB; ++q) put(64 + warp + 8 * q, fx[q][0], fx[q][1]);
    __syncthreads();
#pragma unroll
    for (int q = 0; q < NB; ++q) {
      const int t = warp + 8 * q, kk = 32 * (t & 1), mt = (t >> 1) & 3, nt = t >> 3;
      float acc[NW][4], mag[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
      for (int w = 0; w < NW; ++w) acc[w][0] = acc[w][1] = acc[w][2] = acc[w][3] = 0.0f;
      const uint32_t pa = s_u32(Dg + (16 * mt + (lane & 7) + 8 * ((lane >> 3) & 1)) * kDxK);
      const uint32_t pb = s_u32(Dg + (64 + 8 * nt + (lane & 7)) * kDxK + 8 * (((kk >> 3) + (lane >> 3)) ^ (lane & 7)));
      constexpr int stride = 2 * ROWS_D * kDxK;
      uint32_t fb[P][4];   // both k-steps of each digit of F
#pragma unroll
      for (int p = 0; p < P; ++p) ldsm4(pb + p * stride, fb[p]);
#pragma unroll
      for (int ks = 0; ks < 2; ++ks)
#pragma unroll
        for (int p = 0; p < P; ++p) {
          uint32_t fa[4];
          ldsm4(pa + p * stride + 16 * (((kk >> 3) + 2 * ks + (lane >> 4)) ^ (lane & 7)), fa);
          if (p == 0) mma_abs(mag, fa, fb[0] + 2 * ks);
#pragma unroll
          for (int p2 = 0; p2 < P; ++p2)
            if (p + p2 < NW) mma(acc[(p + p2) % NW], fa, fb[p2] + 2 * ks);
        }
      uint32_t redo = 0;
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const int ea = er[16 * mt + gq + 8 * (e >> 1)], eb = er[64 + 8 * nt + 2 * tq + (e & 1)];
        if (ea == kExpZero || eb == kExpZero) continue;   // a column of zeros
        if (weak(mag[e], 0x1p-6f, LEAD, c[q][e], ea + eb - 4)) {
          redo |= 1u << e;
          continue;
        }
        const int x = ea + eb - 2 * LEAD - 56;
        long long hi = 0, lo = 0;
#pragma unroll
        for (int w = 0; w < 4; ++w) {
          hi = hi * 256 + __float2int_rn(acc[w][e]);
          lo = lo * 256 + __float2int_rn(acc[w + 4][e]);
        }
        if (hi | lo) {   // (hi 2^32 + lo) 2^x
          const double v = fma((double)hi, 4294967296.0, (double)lo);
          if (x > -900 && x < 900) c[q][e] = fma(v, __hiloint2double((x + 1023) << 20, 0), c[q][e]);
          else c[q][e] += ldexp(v, x);
        }
      }
#pragma unroll
      for (int e = 0; e < 4; ++e)
        if (redo >> e & 1) {
          const int o = 16 * mt + gq + 8 * (e >> 1), j = 8 * nt + 2 * tq + (e & 1);
          const int n = (int)imin64(32, K - 64 * ch - kk);
          c[q][e] = dx_dot(raw + (ROWS ? kk * kDxRaw + o : o * kDxRaw + kk), ROWS ? kDxRaw : 1,
                           F + (64 * ch + kk) * fk + j * fj, fk, n, c[q][e]);
        }
    }
  }
  // a non-finite value in this block's range: its products as FP64 FMAs
  if (__syncthreads_or(bad)) {
    for (int i = tid; i < 64 * rp; i += 256) {
      const int64_t o = o0 + (i & 63);
      const int j = i >> 6;
      if (o >= O) continue;
      double t = 0.0;
      for (int64_t k = 64 * c0; k < imin64(K, 64 * c1); ++k)
        t = fma((double)__ldg(X + (ROWS ? o + Nk * k : k + Nk * o)), __ldg(F + k * fk + j * fj), t);
      atomicAdd(C + o * co + j * cj, t);
    }
    return;
  }
#pragma unroll
  for (int q = 0; q < NB; ++q) {
    const int t = warp + 8 * q, mt = (t >> 1) & 3, nt = t >> 3;
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const int64_t o = o0 + 16 * mt + gq + 8 * (e >> 1);
      const int j = 8 * nt + 2 * tq + (e & 1);
      if (o < O && j < rp) atomicAdd(C + o * co + j * cj, c[q][e]);
    }
  }
}
template <int NB, bool ROWS>
cudaError_t launch_dx_gemm_nb(const float* X, int64_t Nk, int64_t Mk, const double* F, int64_t fk, int64_t fj, int rp,
                              double* C, int64_t co, int64_t cj, cudaStream_t st) {
  static bool attr = false;
  if (!attr) {
    const cudaError_t e =
        cudaFuncSetAttribute(dx_gemm_kernel<NB, ROWS>, cudaFuncAttributeMaxDynamicSharedMemorySize, dx_smem(NB));
    if (e != cudaSuccess) return e;
    attr = true;
  }
  const int64_t ob = ((ROWS ? Nk : Mk) + 63) / 64, nch = ((ROWS ? Mk : Nk) + 63) / 64;
  // about four blocks an SM: an output's sums are added once a block
  const int64_t want = std::max<int64_t>(1, std::min<int64_t>(nch, 4LL * device_sm_count() / ob));
  const int64_t chunks = (nch + want - 1) / want;
  count_launch();
  dx_gemm_kernel<NB, ROWS><<<dim3((unsigned)ob, (unsigned)((nch + chunks - 1) / chunks)), 256, dx_smem(NB), st>>>(
      X, Nk, Mk, F, fk, fj, rp, C, co, cj, chunks);
  return cudaGetLastError();
}
template <bool ROWS>
cudaError_t launch_dx_gemm(const float* X, int64_t Nk, int64_t Mk, const double* F, int64_t fk, int64_t fj, int rp,
                           double* C, int64_t co, int64_t cj, cudaStream_t st) {
  if (rp <= 8) return launch_dx_gemm_nb<1, ROWS>(X, Nk, Mk, F, fk, fj, rp, C, co, cj, st);
  if (rp <= 16) return launch_dx_gemm_nb<2, ROWS>(X, Nk, Mk, F, fk, fj, rp, C, co, cj, st);
  if (rp <= 32) return launch_dx_gemm_nb<4, ROWS>(X, Nk, Mk, F, fk, fj, rp, C, co, cj, st);
  return launch_dx_gemm_nb<8, ROWS>(X, Nk, Mk, F, fk, fj, rp, C, co, cj, st);
}

// Z_{k-1}(u, a) = sum_{i, c} Z_k(u + N_{k-1} i, c) G_k(a, i, c): one warp per entry,
// the lanes over (i, c).
__global__ void zdown_kernel(const double* Z, int64_t Np, int64_t nk, int rpc, const double* G, int rpa, double* Zo) {
  const int lane = threadIdx.x & 31;
  const int64_t nwarps = (int64_t)gridDim.x * (blockDim.x >> 5), Nk = Np * nk, len = nk * rpc;
  for (int64_t job = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); job < Np * rpa; job += nwarps) {
    const int64_t u = job % Np;
    const int a = (int)(job / Np);
    double acc = 0.0;
    for (int64_t j = lane; j < len; j += 32) {
      const int64_t i = j % nk, c = j / nk;
      acc = fma(Z[u + Np * i + Nk * c], G[a + (int64_t)rpa * j], acc);   // j = i + n_k c
    }
    acc = warp_sum(acc);
    if (lane == 0) Zo[u + Np * a] = acc;
  }
}

// W_k(c, v) = sum_{a, i} G_k(a, i, c) W_{k-1}(a, i + n_k v): one warp per entry, the
// lanes over (a, i).
__global__ void wup_kernel(const double* Wp, int rpa, int64_t nk, int64_t Mk, const double* G, int rpc, double* Wo) {
  const int lane = threadIdx.x & 31;
  const int64_t nwarps = (int64_t)gridDim.x * (blockDim.x >> 5), len = (int64_t)rpa * nk;
  for (int64_t job = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); job < Mk * rpc; job += nwarps) {
    const int c = (int)(job % rpc);
    const int64_t v = job / rpc;
    double acc = 0.0;
    for (int64_t j = lane; j < len; j += 32) acc = fma(G[j + len * c], Wp[j + len * v], acc);
    acc = warp_sum(acc);
    if (lane == 0) Wo[c + (int64_t)rpc * v] = acc;
  }
}

// dG_k(a, i, c) = sum_v W_{k-1}(a, i + n_k v) Rt_{k+1}(c, v) (Rt = null: one v, 1): one
// warp per entry, the lanes over v.
__global__ void dcore_right_kernel(const double* Wp, int rpa, int64_t nk, int64_t Mk, const double* Rt, int rpc,
                                   double* dG) {
  const int lane = threadIdx.x & 31;
  const int64_t nwarps = (int64_t)gridDim.x * (blockDim.x >> 5), len = (int64_t)rpa * nk;
  for (int64_t job = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); job < len * rpc; job += nwarps) {
    const int64_t ai = job % len;
    const int c = (int)(job / len);
    double acc = 0.0;
    if (Rt == nullptr) {
      if (lane == 0) dG[job] = Wp[ai];
      continue;
    }
    for (int64_t v = lane; v < Mk; v += 32) acc = fma(Wp[ai + len * v], Rt[c + (int64_t)rpc * v], acc);
    acc = warp_sum(acc);
    if (lane == 0) dG[job] = acc;
  }
}

// dG_k(a, i, c) = sum_u L_{k-1}(u, a) Y_k(u + N_{k-1} i, c);  L_0 = [1].
// dG is zeroed first; a warp takes one entry and one chunk of u (lanes split
// the chunk) and adds its sum with an atomic.
__global__ void dcore_kernel(const double* Lp, int64_t Np, int rpa, const double* Y, int64_t nk, int rpc,
                             double* dG, int64_t uc) {
  const int64_t total = (int64_t)rpa * nk * rpc;
  const int64_t Nk = Np * nk;
  if (Lp == nullptr) {
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < total;
         e += (int64_t)gridDim.x * blockDim.x) {
      const int64_t i = (e / rpa) % nk;
      const int c = (int)(e / (rpa * nk));
      dG[e] = Y[i + Nk * c];
    }
    return;
  }
  const int lane = threadIdx.x & 31;
  const int64_t nuc = (Np + uc - 1) / uc;
  const int64_t nwarps = (int64_t)gridDim.x * (blockDim.x >> 5);
  for (int64_t job = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); job < total * nuc; job += nwarps) {
    const int64_t e = job % total, ch = job / total;
    const int a = (int)(e % rpa);
    const int64_t i = (e / rpa) % nk;
    const int c = (int)(e / (rpa * nk));
    const int64_t u0 = ch * uc, u1 = imin64(Np, u0 + uc);
    double acc = 0.0;
    for (int64_t u = u0 + lane; u < u1; u += 32) acc += Lp[u + Np * a] * Y[u + Np * i + Nk * c];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if (lane == 0) atomicAdd(dG + e, acc);
  }
}

int grid_for(int64_t n) {
  return (int)std::max<int64_t>(1, std::min<int64_t>((n + kThreads - 1) / kThreads, 16LL * device_sm_count()));
}

}  // namespace

cudaError_t build_interfaces(const Plan& P, int item, const double* cores, void* ws, cudaStream_t st) {
  const DevItem& it = plan_items_host(&P)[item];
  double* W = (double*)ws;
  const int d = it.d, ds = it.ds;
  for (int k = 1; k <= ds; ++k) {
    const double* Lp = k == 1 ? nullptr : W + it.off_L[k - 1];
    const int64_t n = it.N[k] * it.rpad[k];
    count_launch();
    iface_left_kernel<<<grid_for(n), kThreads, 0, st>>>(Lp, it.N[k - 1], it.rpad[k - 1],
                                                        cores + it.core_off[k], it.n[k - 1],
                                                        it.rpad[k], W + it.off_L[k]);
  }
  for (int k = d; k >= ds + 1; --k) {
    const double* Rn = k == d ? nullptr : W + it.off_Rt[k + 1];
    const int64_t Mn = it.N[d] / it.N[k];
    const int64_t n = (int64_t)it.rpad[k - 1] * it.n[k - 1] * Mn;
    count_launch();
    iface_right_kernel<<<grid_for(n), kThreads, 0, st>>>(Rn, Mn, it.rpad[k], cores + it.core_off[k],
                                                         it.n[k - 1], it.rpad[k - 1], W + it.off_Rt[k]);
  }
  return cudaGetLastError();
}

namespace {

template <int P, int KS, int UT, int NTL, int MODE>
cudaError_t run_expand(expand::ExpandArgs a, cudaStream_t st) {
  a.nub = (a.Nm + UT - 1) / UT;
  // columns per CTA: about eight CTAs per SM, whole staging steps
  const int64_t want = std::max<int64_t>(1, 8LL * device_sm_count() / a.nub);
  a.vlen = ((a.Mm + want - 1) / want + expand::kVT - 1) / expand::kVT * expand::kVT;
  const int64_t ctas = a.nub * ((a.Mm + a.vlen - 1) / a.vlen);
  constexpr int LD = 16 * std::max(KS, 1) + 8, PA = KS ? P : (P + 1) / 2;
  const size_t smem = 2ul * (P * UT + PA * expand::kVT) * LD + sizeof(int) * (2 * UT + expand::kVT);
  auto k = expand::expand_kernel<P, KS, UT, NTL, MODE>;
  static bool attr = false;
  if (!attr) {
    const cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    attr = true;
  }
  count_launch();
  k<<<(unsigned)ctas, expand::kThreads, smem, st>>>(a);
  return cudaGetLastError();
}
template <int P, int NTL, int MODE>
cudaError_t run_expand_ks(const expand::ExpandArgs& a, cudaStream_t st) {
  if (a.rp <= 8) return run_expand<P, 0, 256, NTL, MODE>(a, st);
  // rows that leave two CTAs an SM in shared memory, as far as 64
  switch ((a.rp + 15) / 16) {
    case 1: return run_expand<P, 1, P == 7 ? 256 : 128, NTL, MODE>(a, st);
    case 2: return run_expand<P, 2, P == 7 ? 128 : 64, NTL, MODE>(a, st);
    case 3: return run_expand<P, 3, 128, NTL, MODE>(a, st);
    default: return run_expand<P, 4, 128, NTL, MODE>(a, st);
  }
}

// out2 = the sums of the kErrSlots pairs of slots.
__global__ void err_slots_kernel(const double* slots, double* out2) {
  static_assert(expand::kErrSlots == 64, "two pairs a lane");
  double a = slots[2 * threadIdx.x] + slots[2 * threadIdx.x + 64];   // pairs lane, lane + 32
  double b = slots[2 * threadIdx.x + 1] + slots[2 * threadIdx.x + 65];
  a = warp_sum(a);
  b = warp_sum(b);
  if (threadIdx.x == 0) out2[0] = a, out2[1] = b;
}

}  // namespace

cudaError_t launch_reconstruct(const Plan& P, int item, const double* cores, void* Xt, int x_f64,
                               const void* Xcmp, int cmp_f64, double* out2, void* ws,
                               cudaStream_t st) {
  const DevItem& it = plan_items_host(&P)[item];
  cudaError_t e = build_interfaces(P, item, cores, ws, st);
  if (e != cudaSuccess) return e;
  if (out2) {
    e = cudaMemsetAsync(out2, 0, 2 * sizeof(double), st);
    if (e != cudaSuccess) return e;
  }
  double* W = (double*)ws;
  const int ds = it.ds;
  const int64_t Nm = it.N[ds], Mm = it.N[it.d] / it.N[ds];
  // Digit arithmetic (expand.cuh) for FP32 data from 3 2^18 entries on, with both
  // interfaces at least as long as a staging step and enough FP64 products to spare, entries x
  // rank: 3 2^21 for the output, 3 2^20 for the error sums.  Measured (whole call, us, FP64
  // kernel -> digit kernel): output, below the line 900 x 900 rank 3 18.5 -> 22.8, 1000 x 1000 rank 3
  // 19.9 -> 23.3, 93^3 rank 2 20.7 -> 27.1; above it 900 x 900 rank 8 24.8 -> 22.8, 30^4 rank 8 33.0 ->
  // 31.1, 128^3 rank 10 58 -> 33, 200^3 rank 2 62 -> 42, rank 24 385 -> 131, 256^4 rank 6 51300 -> 8880
  // (4770 with five digits, which left entries far below their row's and column's scale without
  // correct bits; 16 warps an SM wait on their own chains, half of the issue slots used).
  // Error sums, below 900 x 900 rank 1 35.1 -> 36.1, 93^3 rank 2 39.4 -> 40.1; above 64 x 12500 rank 4
  // 39.1 -> 32.6, 30^4 rank 8 52 -> 44, 200^3 rank 2 117 -> 74, 24^6 rank 10 4590 -> 1117 (923 with
  // seven digits and residuals in FP32 pairs, which were further off than FP64 ones).
  const int64_t entries = Nm * Mm;
  if ((Xt ? !x_f64 : !cmp_f64) && Nm >= 64 && Mm >= 64 && entries >= (3 << 18) &&
      entries * it.rpad[ds] >= (Xt ? 3 << 21 : 3 << 20)) {
    expand::ExpandArgs a;
    a.L = W + it.off_L[ds];
    a.Rt = W + it.off_Rt[ds + 1];
    a.Nm = Nm;
    a.Mm = Mm;
    a.rp = it.rpad[ds];
    a.out = (float*)Xt;
    a.X = (const float*)Xcmp;
    a.out2 = out2;
    a.vec = Nm % 4 == 0 && ((uintptr_t)(Xt ? Xt : Xcmp) & 15) == 0 ? 1 : 0;
    a.slots = 0;
    if (Xt) return run_expand_ks<7, 2, 0>(a, st);
    if (it.off_small == 0) return run_expand_ks<8, 2, 1>(a, st);   // (a batched plan of one has no such scratch)
    a.out2 = W + it.off_small;
    a.slots = 1;
    e = cudaMemsetAsync(a.out2, 0, 2 * expand::kErrSlots * sizeof(double), st);
    if (e == cudaSuccess) e = run_expand_ks<8, 2, 1>(a, st);
    if (e != cudaSuccess) return e;
    count_launch();
    err_slots_kernel<<<1, 32, 0, st>>>(a.out2, out2);
    return cudaGetLastError();
  }
  count_launch();
  dense_kernel<<<grid_for(Nm * Mm), kThreads, 0, st>>>(W + it.off_L[ds], W + it.off_Rt[ds + 1], Nm, Mm,
                                                       it.rpad[ds], Xt, x_f64, Xcmp, cmp_f64, out2);
  return cudaGetLastError();
}

// Adjoint of the reconstruction: for every core k,
//   dG_k(a, i, c) = sum_{u, v} L_{k-1}(u, a) dX(u + N_{k-1} i + N_k v) Rt_{k+1}(c, v)
// with the left / right interfaces of the train.  dX is contracted twice, at the
// middle: Z_ds = dX Rt_{ds+1}^T for the cores up to ds, W_ds = L_ds^T dX for the
// others; from there the cores absorb one mode at a time (Z_{k-1} from Z_k and G_k,
// W_k from W_{k-1} and G_k), so only these two products see every entry (2 N r
// FMAs).  One contraction per core (d N r FMAs, and the interfaces of length
// N_{d-1}) took 4.5 ms for 32^5 of rank 8; this takes 1.2 ms with the two products on the
// FP64 pipe and 0.76 with them in digit arithmetic.
cudaError_t launch_reconstruct_backward(const Plan& P, int item, const double* cores, const void* dXt,
                                        int dx_f64, double* dcores, void* ws, cudaStream_t st) {
  const DevItem& it = plan_items_host(&P)[item];
  double* W = (double*)ws;
  const int d = it.d, ds = it.ds;
  cudaError_t e = build_interfaces(P, item, cores, ws, st);
  if (e != cudaSuccess) return e;
  static bool attr = false;
  if (!attr) {
    e = cudaFuncSetAttribute(ygram_kernel<64>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             4 * 64 * 32 * (int)sizeof(double));
    if (e != cudaSuccess) return e;
    attr = true;
  }
  const int64_t Nm = it.N[ds], Mm = it.N[d] / Nm;
  const int rp = it.rpad[ds];
  const int64_t sms = device_sm_count();
  const bool dig = !dx_f64 && Nm >= 64 && Mm >= 64 && Nm * Mm >= kDxMin && (Nm + 63) / 64 < (1LL << 31) &&
                     (Mm + 63) / 64 < (1LL << 31);
  {  // Z_ds = dX Rt_{ds+1}^T; v chunks sized so that about 32k warp jobs cover the entries
    double* Z = W + it.off_Z[ds];
    e = cudaMemsetAsync(Z, 0, sizeof(double) * Nm * rp, st);
    if (e != cudaSuccess) return e;
    const int64_t vc = std::max<int64_t>(16, (Nm * Mm) / (32LL * 32768));
    const int64_t nrb = (Nm + 31) / 32, nvg = ((Mm + vc - 1) / vc + 3) / 4;
    const int g = (int)std::max<int64_t>(1, std::min<int64_t>(nrb * nvg, 16 * sms));
    const double* Rt = W + it.off_Rt[ds + 1];
    if (dig) {
      e = launch_dx_gemm<true>((const float*)dXt, Nm, Mm, Rt, rp, 1, rp, Z, 1, Nm, st);
      if (e != cudaSuccess) return e;
    } else {
      count_launch();
      if (rp <= 8)
        ygram_kernel<8><<<g, 128, 4 * 8 * 32 * sizeof(double), st>>>(dXt, dx_f64, Nm, Mm, Rt, rp, Z, vc);
      else if (rp <= 16)
        ygram_kernel<16><<<g, 128, 4 * 16 * 32 * sizeof(double), st>>>(dXt, dx_f64, Nm, Mm, Rt, rp, Z, vc);
      else if (rp <= 32)
        ygram_kernel<32><<<g, 128, 4 * 32 * 32 * sizeof(double), st>>>(dXt, dx_f64, Nm, Mm, Rt, rp, Z, vc);
      else
        ygram_kernel<64><<<g, 128, 4 * 64 * 32 * sizeof(double), st>>>(dXt, dx_f64, Nm, Mm, Rt, rp, Z, vc);
    }
  }
  {  // W_ds = L_ds^T dX; row chunks likewise
    double* Wd = W + it.off_Wd[ds];
    e = cudaMemsetAsync(Wd, 0, sizeof(double) * Mm * rp, st);
    if (e != cudaSuccess) return e;
    const int V = rp <= 8 ? 4 : rp <= 16 ? 2 : 1;
    const int64_t nvg = (Mm + V - 1) / V;
    const int64_t want = std::max<int64_t>(1, 64 * sms / nvg);
    const int64_t uc = std::max<int64_t>(256, (Nm + want - 1) / want);
    const int64_t jobs = nvg * ((Nm + uc - 1) / uc);
    const int g = (int)std::max<int64_t>(1, std::min<int64_t>((jobs + 3) / 4, 16 * sms));
    const double* L = W + it.off_L[ds];
    if (dig) {
      e = launch_dx_gemm<false>((const float*)dXt, Nm, Mm, L, 1, Nm, rp, Wd, rp, 1, st);
      if (e != cudaSuccess) return e;
    } else {
      count_launch();
      if (rp <= 8) wgram_kernel<8, 4><<<g, 128, 0, st>>>(dXt, dx_f64, Nm, Mm, L, rp, Wd, uc);
      else if (rp <= 16) wgram_kernel<16, 2><<<g, 128, 0, st>>>(dXt, dx_f64, Nm, Mm, L, rp, Wd, uc);
      else if (rp <= 32) wgram_kernel<32, 1><<<g, 128, 0, st>>>(dXt, dx_f64, Nm, Mm, L, rp, Wd, uc);
      else wgram_kernel<64, 1><<<g, 128, 0, st>>>(dXt, dx_f64, Nm, Mm, L, rp, Wd, uc);
    }
  }
  for (int k = ds; k >= 1; --k) {
    const int64_t Np = it.N[k - 1], nk = it.n[k - 1];
    const int rpa = it.rpad[k - 1], rpc = it.rpad[k];
    const int64_t nout = (int64_t)rpa * nk * rpc;
    e = cudaMemsetAsync(dcores + it.core_off[k], 0, sizeof(double) * nout, st);
    if (e != cudaSuccess) return e;
    const int64_t uc = std::max<int64_t>(256, (nout * Np) / 32768);
    count_launch();
    dcore_kernel<<<grid_for(nout * ((Np + uc - 1) / uc) * 32), kThreads, 0, st>>>(
        k == 1 ? nullptr : W + it.off_L[k - 1], Np, rpa, W + it.off_Z[k], nk, rpc, dcores + it.core_off[k], uc);
    if (k > 1) {
      count_launch();
      zdown_kernel<<<grid_for(Np * rpa * 32), kThreads, 0, st>>>(W + it.off_Z[k], Np, nk, rpc, cores + it.core_off[k],
                                                                rpa, W + it.off_Z[k - 1]);
    }
  }
  for (int k = ds + 1; k <= d; ++k) {
    const int64_t nk = it.n[k - 1], Mk = it.N[d] / it.N[k];
    const int rpa = it.rpad[k - 1], rpc = it.rpad[k];
    count_launch();
    dcore_right_kernel<<<grid_for((int64_t)rpa * nk * rpc * 32), kThreads, 0, st>>>(
        W + it.off_Wd[k - 1], rpa, nk, Mk, k == d ? nullptr : W + it.off_Rt[k + 1], rpc, dcores + it.core_off[k]);
    if (k < d) {
      count_launch();
      wup_kernel<<<grid_for(Mk * rpc * 32), kThreads, 0, st>>>(W + it.off_Wd[k - 1], rpa, nk, Mk,
                                                              cores + it.core_off[k], rpc, W + it.off_Wd[k]);
    }
  }
  return cudaGetLastError();
}

}  // namespace tts
