// The dense product X~(u, v) = sum_c L(u, c) Rt(c, v) of the two interfaces in
// digit arithmetic on the tensor cores: FP32 output, or the error sums against
// an FP32 tensor.
//
// What bounded the FP64 form: a warp's FP64 FMA holds its sub-partition for 64
// cycles on this GPU (1.72 FMA per cycle and SM measured), so rank 6 cost 51 ms
// for 256^4 entries where writing them takes 2.5 ms.  Here every FP64 value is
// written in P balanced base-256 digits, P = 7 for the output and 8 for the error sums: 8 P -
// 3 bits (one less at ranks above 48) below the scale of its row or column; the digits are exact BF16 values, a product of two
// digits summed over a contraction of up to 64 and over the pairs of equal weight stays
// below 2^23, so the FP32 accumulation of mma.sync is exact.  (Splitting operands so
// that low-precision products sum without error: Ozaki, Ogita, Oishi, Rump, Numer.
// Algorithms 59, 2012.)  Pairs (i, j) with i + j < P are kept (P (P + 1) / 2 MMAs per
// k-step), one accumulator per weight, and the result is put together by Horner's rule.
//
// Scales (powers of two): per column c of the CTA's rows of L (moved over to the
// rows of Rt, so that no gauge between the two costs digits), then per row u of L
// and per column v of Rt.  In units of the largest term that any entry of the row and
// the column could have, a term is off at P = 7 by at most 2^-53 (two roundings of 2^-54)
// plus the pairs left out, 6 2^14 2^-56 2^-10 and smaller ones: 2^-49.2 in all (2^-47.2 at
// ranks above 48; in the accumulators' units 2^-31.2 either way); at P = 8 by 2^-57.1
// (2^-55.1).
//
// FP32 output: an entry below 2^27 times that bound, or below sixteen times what the last
// addition rounds off, is summed again in FP64 (dot64).  So every entry is within 1/4 of a
// half-ulp of the FP64 sum rounded once, however far it lies below its row's and column's
// scale -- localised components that are large in different places, cancellation.
// For random factors one entry in 10^4 is summed again; where all are (components that
// nowhere meet) the call costs what the FP64 form did and the digits besides (4000 x 4000,
// rank 16: 86 us for random factors, 625 for such, 467 in FP64 throughout).
//
// Error sums: a residual is x minus the three-word sum of the weights, squares and sums are
// held in words of their own (below), so that neither the residuals nor the sums are further
// off than in FP64: 1009 x 803, sum of squares 1e-16 off at most (FP64 2e-15), a tensor met
// to rounding 1e-16 as in FP64.
#pragma once
#include <cstdint>

#include "digits.cuh"
#include "internal.cuh"

namespace tts {
namespace expand {

using namespace digit;

constexpr int kThreads = 256, kWarps = 8;
constexpr int kVT = 64;          // columns v staged at a time

struct ExpandArgs {
  const double *L, *Rt;
  int64_t Nm, Mm;
  int rp;
  int64_t nub, vlen;   // blocks of u, columns v per CTA
  float* out;          // FP32 output
  const float* X;      // or the tensor to compare with
  double* out2;        // [2], added to with atomics, or kErrSlots pairs of it (slots)
  int slots;
  int vec;             // float4 accesses are aligned
};

__device__ __forceinline__ float pow2f(int e) {  // 2^e, zero below the normal range, e <= 127
  return e < -126 ? 0.0f : __int_as_float((min(e, 127) + 127) << 23);
}

// A thousand CTAs' error sums added into one FP64 word one after another drift (the
// addends are alike: 1.4e-15 of the sum); they go to this many pairs first.
constexpr int kErrSlots = 64;

__device__ __forceinline__ void two_sum(float a, float b, float& s, float& e) {
  s = __fadd_rn(a, b);
  const float bb = __fsub_rn(s, a);
  e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
}

// An entry in FP64.
__device__ __noinline__ double dot64(const double* L, int64_t ldl, const double* R, int rp) {
  double s = 0.0;
  for (int c = 0; c < rp; ++c) s = fma(__ldg(L + ldl * c), __ldg(R + c), s);
  return s;
}

// KS k-steps of 16 (rp <= 16 KS; KS = 0: rp <= 8, one k-step holds two digits),
// UT rows u per CTA, NTL n-tiles of 8 u a warp takes at a time.  MODE 0: FP32
// output; 1: error sums.
//
// KS = 0: a k-step of 16 takes two pairs of equal weight at once, [digit 2m, digit
// 2m + 1] of Rt against [digit j, digit j - 1] of L (weights 2m + j): 16 MMAs instead of
// 28 (P = 7), 20 instead of 36 (P = 8).
template <int P, int KS, int UT, int NTL, int MODE>
__global__ void __launch_bounds__(kThreads, KS <= 2 ? 2 : 1) expand_kernel(const ExpandArgs a) {
  constexpr bool HALF = KS == 0;
  constexpr int KN = HALF ? 1 : KS, K = 16 * KN, LD = K + 8;   // a row's words (an odd number of 16-byte chunks)
  constexpr int PA = HALF ? (P + 1) / 2 : P;                   // digit arrays of Rt
  // The leading digit's full scale 2^LEAD is set so that A0 256 + A1, the sums of
  // the two largest weights, is an exact FP32 integer for every rank of the
  // instance: rp (2^(2 LEAD + 8) + 2^(LEAD + 8)) <= 2^24.
  constexpr int LEAD = KS == 4 ? 4 : 5, B = 8 * (P - 1) + LEAD;
  constexpr int UW = 8 * NTL, GU = UT / UW;   // a warp's u, groups of them
  extern __shared__ __align__(16) unsigned char sm[];
  uint16_t* Ld = reinterpret_cast<uint16_t*>(sm);                 // [P][UT][LD]
  uint16_t* Rd = Ld + (size_t)P * UT * LD;                        // [PA][kVT][LD]
  int* eu = reinterpret_cast<int*>(Rd + (size_t)PA * kVT * LD);   // [UT]
  int* ev = eu + UT;                                              // [kVT]
  float* fu = reinterpret_cast<float*>(ev + kVT);                 // [UT] 2^(eu - eU)
  __shared__ int ec[64];
  __shared__ int eU, eLow;   // largest and smallest row exponent
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g = lane >> 2, t = lane & 3;
  const int64_t ub = blockIdx.x % a.nub, vb = blockIdx.x / a.nub;
  const int64_t u0 = ub * UT, v0 = vb * a.vlen, v1 = imin64(a.Mm, v0 + a.vlen);
  const int nu = (int)imin64(UT, a.Nm - u0);
  double e2 = 0.0, x2 = 0.0;
  // Column n of n-tile nt is u = (UW / 4) (n / 2) + 2 nt + n % 2 of the warp's
  // group, so that a lane's results are consecutive in u; the rows of a tile
  // lie together in shared memory (ldmatrix without bank conflicts).
  auto row_of = [](int i) {
    const int k = i & (UW - 1), nt = (k >> 1) & (NTL - 1), n = 2 * (k / (2 * NTL)) + (k & 1);
    return i - k + 8 * nt + n;
  };

  // ---- the rows of L: column exponents, row exponents, digits
  if (tid < 64) ec[tid] = kExpZero;
  if (tid == 0) eU = kExpZero, eLow = -kExpZero;
  __syncthreads();
  int bad = 0;
  for (int c = warp; c < a.rp; c += kWarps) {
    int m = kExpZero;
    for (int i = lane; i < nu; i += 32) {
      const double x = a.L[u0 + i + a.Nm * c];
      bad |= undigital(x) ? 1 : 0;
      m = max(m, exp_of(x));
    }
    m = __reduce_max_sync(0xffffffffu, m);
    if (lane == 0) ec[c] = m;
  }
  __syncthreads();
  for (int i = tid; i < UT; i += kThreads) {
    int m = kExpZero;
    if (i < nu)
      for (int c = 0; c < a.rp; ++c) {
        const int e = exp_of(a.L[u0 + i + a.Nm * c]);
        if (e != kExpZero) m = max(m, e - ec[c]);
      }
    eu[i] = m;
    if (m != kExpZero) atomicMax(&eU, m), atomicMin(&eLow, m);
    for (int c2 = 0; c2 < (HALF ? 4 : K / 2); ++c2) {
      uint32_t d0[P], d1[P];
      const int c = 2 * c2;
      const double xa = i < nu && c < a.rp ? a.L[u0 + i + a.Nm * c] : 0.0;
      const double xb = i < nu && c + 1 < a.rp ? a.L[u0 + i + a.Nm * (c + 1)] : 0.0;
      digits<P>(fixed<B>(xa, m + (c < a.rp ? ec[c] : 0)), d0);
      digits<P>(fixed<B>(xb, m + (c + 1 < a.rp ? ec[c + 1] : 0)), d1);
#pragma unroll
      for (int p = 0; p < P; ++p) {
        uint16_t* w = Ld + ((size_t)p * UT + row_of(i)) * LD + c;
        *reinterpret_cast<uint32_t*>(w) = d0[p] | (d1[p] << 16);
        if constexpr (HALF) *reinterpret_cast<uint32_t*>(w + 8) = p ? d0[p - 1] | (d1[p - 1] << 16) : 0u;
      }
    }
  }
  // contraction padding of the columns' digits (never written again)
  for (int o = tid; o < PA * kVT * LD / 2; o += kThreads) reinterpret_cast<uint32_t*>(Rd)[o] = 0u;
  const bool bad_l = __syncthreads_or(bad);
  for (int i = tid; i < UT; i += kThreads) fu[i] = eu[i] == kExpZero ? 0.0f : pow2f(eu[i] - eU);
  // rows within 2^60 of one another: products with fu are exact
  const bool narrow = eU - eLow <= 60;

  // Error sums, scaled by 2^(-2 kb): the sum, the rounding errors of its additions, those
  // of the squares and those of the latter's additions.  (The trailing bits of squares are
  // not evenly spread, and dl^2 below is always positive: without the last word a sum is
  // 5e-16 too small.)
  float s_e = 0.f, s_el = 0.f, s_er = 0.f, s_eq = 0.f, s_x = 0.f, s_xl = 0.f, s_xr = 0.f, s_xq = 0.f;
  int kb = -100;
  // into the FP64 sums (a sum that is not finite keeps its leading part only)
  auto fold = [&]() {
    const double sc = __hiloint2double((2 * kb + 1023) << 20, 0);
    e2 += (fabsf(s_e) <= 3.0e38f ? (double)s_e + ((double)s_el + ((double)s_er + (double)s_eq)) : (double)s_e) * sc;
    x2 += (fabsf(s_x) <= 3.0e38f ? (double)s_x + ((double)s_xl + ((double)s_xr + (double)s_xq)) : (double)s_x) * sc;
    s_e = s_el = s_er = s_eq = s_x = s_xl = s_xr = s_xq = 0.f;
  };
  for (int64_t vc = v0; vc < v1; vc += kVT) {
    const int nv = (int)imin64(kVT, v1 - vc);
    if (MODE == 1) fold();   // the FP32-pair sums stay short
    __syncthreads();
    // ---- columns vc.. of Rt: four threads a column
    bad = 0;
    bool low = false, ordinary = false;   // error sums: X~ below 2^-160, or not
    {
      const int v = tid >> 2, q = tid & 3;
      const double* r = a.Rt + (vc + v) * a.rp;
      int m = kExpZero;
      if (v < nv)
        for (int c = q; c < a.rp; c += 4) {
          const double x = r[c];
          bad |= undigital(x) ? 1 : 0;
          const int e = exp_of(x);
          if (e != kExpZero && ec[c] != kExpZero) m = max(m, e + ec[c]);
        }
      m = max(m, __shfl_xor_sync(0xffffffffu, m, 1));
      m = max(m, __shfl_xor_sync(0xffffffffu, m, 2));
      if (q == 0) ev[v] = m;
      if (MODE == 1 && m != kExpZero && eU != kExpZero) {
        bad |= m + eU > 110 ? 1 : 0;   // X~ past FP32's range
        low = m + eU < -160;
        ordinary = !low;
      }
      for (int c = 2 * q; c < a.rp; c += 8) {
        uint32_t d0[P], d1[P];
        // a zero column of L has no terms: its entries of Rt count as zero
        const double xa = v < nv && ec[c] != kExpZero ? r[c] : 0.0;
        const double xb = v < nv && c + 1 < a.rp && ec[c + 1] != kExpZero ? r[c + 1] : 0.0;
        digits<P>(fixed<B>(xa, m - ec[c]), d0);
        digits<P>(fixed<B>(xb, m - ec[min(c + 1, 63)]), d1);
#pragma unroll
        for (int p = 0; p < P; ++p)
          *reinterpret_cast<uint32_t*>(Rd + ((size_t)(HALF ? p / 2 : p) * kVT + v) * LD + (HALF ? 8 * (p & 1) : 0) + c) =
              d0[p] | (d1[p] << 16);
      }
    }
    bool slow = __syncthreads_or(bad) || bad_l;
    if (MODE == 1 && __syncthreads_or(low)) slow |= !__syncthreads_or(ordinary);
    if (slow) {  // a non-finite or subnormal factor, X~ out of range: FP64 arithmetic as it stands
      for (int o = tid; o < nu * nv; o += kThreads) {
        const int64_t u = u0 + o % nu, v = vc + o / nu;
        const double s = dot64(a.L + u, a.Nm, a.Rt + v * a.rp, a.rp);
        if constexpr (MODE == 0) {
          a.out[u + a.Nm * v] = (float)s;
        } else {
          const double x = (double)a.X[u + a.Nm * v];
          e2 += (x - s) * (x - s);
          x2 += x * x;
        }
      }
      continue;
    }
    // ---- products: a warp takes UW rows u and all its column steps of 16
    for (int job = warp; job < GU * (kVT / 16); job += kWarps) {
      const int gu = job % GU, vs = (job / GU) * 16;
      if (vs >= nv || gu * UW >= nu) continue;
      float xv[2][2 * NTL];   // the lane's entries of X, loaded ahead of the products
      if constexpr (MODE == 1) {
        const int ur = gu * UW + 2 * NTL * t;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int v = vs + g + 8 * h;
          const float* p = a.X + u0 + ur + a.Nm * (vc + v);
          if (a.vec && ur + 2 * NTL <= nu && v < nv) {
#pragma unroll
            for (int n = 0; n < NTL; n += 2) {
              const float4 w = __ldcs(reinterpret_cast<const float4*>(p + 2 * n));
              xv[h][2 * n] = w.x, xv[h][2 * n + 1] = w.y, xv[h][2 * n + 2] = w.z, xv[h][2 * n + 3] = w.w;
            }
          } else {
#pragma unroll
            for (int n = 0; n < 2 * NTL; ++n) xv[h][n] = ur + n < nu && v < nv ? __ldg(p + n) : 0.0f;
          }
        }
      }
      float acc[NTL][P][4];
      const uint32_t ra = s_u32(Rd + (vs + (lane & 7) + 8 * ((lane >> 3) & 1)) * LD + 8 * (lane >> 4));
      const uint32_t la = s_u32(Ld + (gu * UW + 8 * (lane >> 4) + (lane & 7)) * LD + 8 * ((lane >> 3) & 1));
#pragma unroll
      for (int ks = 0; ks < KN; ++ks) {
        uint32_t fa[PA][4];
#pragma unroll
        for (int i = 0; i < PA; ++i) ldsm4(ra + 2 * (i * kVT * LD + 16 * ks), fa[i]);
#pragma unroll
        for (int j = 0; j < P; ++j) {
          uint32_t fb[NTL][2];
#pragma unroll
          for (int n = 0; n < NTL; n += 2) {
            uint32_t b[4];
            ldsm4(la + 2 * (j * UT * LD + 8 * n * LD + 16 * ks), b);
            fb[n][0] = b[0], fb[n][1] = b[1], fb[n + 1][0] = b[2], fb[n + 1][1] = b[3];
          }
#pragma unroll
          for (int i = 0; i < PA; ++i)
            if ((HALF ? 2 * i : i) + j < P)
#pragma unroll
              for (int n = 0; n < NTL; ++n) {
                float* c = acc[n][((HALF ? 2 * i : i) + j) % P];
                if (ks == 0 && j <= (HALF ? 1 : 0)) mma0(c, fa[i], fb[n]);   // the first pair of its weight
                else mma(c, fa[i], fb[n]);
              }
        }
      }
      constexpr float kD = 0x1p-8f;
      const float least = 0.0625f * (float)a.rp;
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int v = vs + g + 8 * h;
        if (v >= nv) continue;
        const int ur = gu * UW + 2 * NTL * t;   // this lane's 2 NTL consecutive rows
        const int64_t at = u0 + ur + a.Nm * (vc + v);
        const int e_v = ev[v];
        if constexpr (MODE == 0) {
          float r[2 * NTL];
          uint32_t redo = 0;   // entries too small for their digits
#pragma unroll
          for (int n = 0; n < NTL; ++n)
#pragma unroll
            for (int e = 0; e < 2; ++e) {
              // (A0 256 + A1) + 2^-8 A2 = x + xe without error (the first sum is an exact
              // integer and the second a multiple of 2^-8 below 2^16 wherever it is the larger),
              // then the rest y in one rounding each
              const int q = 2 * h + e;
              float s = acc[n][P - 1][q];
#pragma unroll
              for (int w = P - 2; w >= 3; --w) s = fmaf(s, kD, acc[n][w][q]);
              const float a01 = fmaf(acc[n][0][q], 256.0f, acc[n][1][q]);
              const float x = fmaf(acc[n][2][q], kD, a01);
              const float xe = fmaf(acc[n][2][q], kD, a01 - x);
              const float y = fmaf(s, 0x1p-16f, xe);
              r[2 * n + e] = x + y;
              if (fabsf(r[2 * n + e]) < fmaf(fabsf(y), 16.0f, least)) redo |= 1u << (2 * n + e);
            }
          // times 2^(eu + ev) over full scale
          const int eb = eU + e_v - 2 * LEAD - 8;
          if (narrow && eb >= -100 && eb <= 120) {
            const float gv = pow2f(eb);
#pragma unroll
            for (int n = 0; n < 2 * NTL; ++n) r[n] = r[n] * fu[ur + n] * gv;
          } else {
#pragma unroll
            for (int n = 0; n < 2 * NTL; ++n) {
              const int x = eu[ur + n] + e_v - 2 * LEAD - 8;
              const int x1 = max(min(x, 126), -126), x2 = max(min(x - x1, 126), -126);
              r[n] = r[n] * pow2f(x1) * pow2f(x2);
            }
          }
          // (a zero row or column has no terms)
          if (redo && e_v != kExpZero)
#pragma unroll 1
            for (; redo; redo &= redo - 1) {
              const int k = __ffs(redo) - 1;
              if (ur + k >= nu || eu[ur + k] == kExpZero) continue;
              const float s = (float)dot64(a.L + u0 + ur + k, a.Nm, a.Rt + (vc + v) * a.rp, a.rp);
#pragma unroll
              for (int n = 0; n < 2 * NTL; ++n) r[n] = n == k ? s : r[n];
            }
          if (a.vec && ur + 2 * NTL <= nu) {
#pragma unroll
            for (int n = 0; n < NTL; n += 2)
              __stcs(reinterpret_cast<float4*>(a.out + at + 2 * n),
                     make_float4(r[2 * n], r[2 * n + 1], r[2 * n + 2], r[2 * n + 3]));
          } else {
#pragma unroll
            for (int n = 0; n < 2 * NTL; ++n)
              if (ur + n < nu) a.out[at + n] = r[n];
          }
        } else {
          float hi[2 * NTL], mid[2 * NTL], lo[2 * NTL];
          const float(&x)[2 * NTL] = xv[h];
          float mx = 0.f, mt = 0.f;
#pragma unroll
          for (int n = 0; n < NTL; ++n)
#pragma unroll
            for (int e = 0; e < 2; ++e) {
              const int k = 2 * n + e, q = 2 * h + e;
              // (A0 256 + A1) + 2^-8 A2 = hi + r as above and r + 2^-16 A3 = t, a multiple of
              // 2^-16 below 2^7, exactly; t + 2^-24 A4 = mid + lo, then the rest
              const float a01 = fmaf(acc[n][0][q], 256.0f, acc[n][1][q]);
              hi[k] = fmaf(acc[n][2][q], kD, a01);
              const float t = fmaf(acc[n][3][q], 0x1p-16f, fmaf(acc[n][2][q], kD, a01 - hi[k]));
              float s = acc[n][P - 1][q];
#pragma unroll
              for (int w = P - 2; w >= 5; --w) s = fmaf(s, kD, acc[n][w][q]);
              mid[k] = fmaf(acc[n][4][q], 0x1p-24f, t);
              lo[k] = fmaf(s, 0x1p-32f, fmaf(acc[n][4][q], 0x1p-24f, t - mid[k]));
              // (fu is zero for a row past the block, whose x is zero, too)
              mx = fmaxf(mx, fabsf(x[k]));
              mt = fmaxf(mt, fabsf(hi[k] * fu[ur + k]));
            }
          // running scale 2^kb of the sums: at least this batch's largest value
          const int eb = eU + e_v - 2 * LEAD - 8;
          int k2 = max(kb, (int)(__float_as_uint(mx) >> 23) - 126);
          if (mt > 0.f) k2 = max(k2, (int)(__float_as_uint(mt) >> 23) - 126 + eb);
          k2 = min(k2, 126);
          if (k2 != kb) {
            const float f = pow2f(max(2 * (kb - k2), -126));
            s_e *= f, s_el *= f, s_er *= f, s_eq *= f, s_x *= f, s_xl *= f, s_xr *= f, s_xq *= f;
            kb = k2;
          }
          const float fx = pow2f(-kb), ft = pow2f(min(eb - kb, 127));
#pragma unroll
          for (int k = 0; k < 2 * NTL; ++k) {
            // x - hi - mid - lo = d + dl, d the leading 24 bits
            const float xs = x[k] * fx, f = fu[ur + k] * ft;
            float d, dl, el;
            two_sum(xs, -(hi[k] * f), d, dl);
            if (fabsf(d) <= 3.0e38f) {   // an infinite entry stays infinite
              two_sum(d, -(mid[k] * f), d, el);
              dl += fmaf(-lo[k], f, el);
              const float s = __fadd_rn(d, dl);
              dl = __fsub_rn(dl, __fsub_rn(s, d));
              d = s;
            } else {
              dl = 0.f;
            }
            const float p = __fmul_rn(d, d);
            const float pe = fmaf(2.0f * d, dl, __fmaf_rn(d, d, -p));   // and dl^2, below its last bit
            float s, c;
            two_sum(s_e, p, s, c);
            s_e = s;
            s_el += c;
            s = __fadd_rn(s_er, pe);
            s_eq = fmaf(dl, dl, __fadd_rn(s_eq, __fsub_rn(pe, __fsub_rn(s, s_er))));
            s_er = s;
            const float px = __fmul_rn(xs, xs), pxe = __fmaf_rn(xs, xs, -px);
            two_sum(s_x, px, s, c);
            s_x = s;
            s_xl += c;
            s = __fadd_rn(s_xr, pxe);
            s_xq += __fsub_rn(pxe, __fsub_rn(s, s_xr));
            s_xr = s;
          }
        }
      }
    }
  }
  if constexpr (MODE == 1) {
    fold();
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      e2 += __shfl_xor_sync(0xffffffffu, e2, o);
      x2 += __shfl_xor_sync(0xffffffffu, x2, o);
    }
    __shared__ double red[2][kWarps];
    if (lane == 0) red[0][warp] = e2, red[1][warp] = x2;
    __syncthreads();
    if (tid < 2) {
      double s = 0.0;
      for (int w = 0; w < kWarps; ++w) s += red[tid][w];
      atomicAdd(a.out2 + (a.slots ? 2 * (blockIdx.x % kErrSlots) : 0u) + tid, s);
    }
  }
}

}  // namespace expand
}  // namespace tts
