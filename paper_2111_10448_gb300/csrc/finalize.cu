// FP64 finalize: orthonormal bases, ranks, the one-pass middle core and the
// core products (Sec. 3.2; Algorithm 2 steps 4-8; eq. (3.1) and its row-space
// mirror; eq. (3.3) for the middle core).
//
// Bases.  The paper takes a CPQR of each sketch and keeps Q(:, 1:r_k); it
// forms the ON bases of the distributed sketches with a skinny (TSQR) QR
// (Sec. 4.2, Benson et al.).  Here every basis sketch Y (m x l, m up to
// n^{ceil(d/2)}) is reduced by a TSQR tree of Householder QRs of row blocks;
// the CPQR is taken on the l x l root factor R, which has the same column
// norms and inner products as Y (Y = Q_1 R), so it selects the same pivots:
// R Pi = Q_2 Rt.  Then Q_k = Q_1 Q_2(:, 1:r_k), formed top-down through the
// tree.  Signs are normalised so that diag(Rt) >= 0.
//
// Ranks.  Fixed-rank mode keeps the (clamped) target.  Tolerance mode takes
// the smallest r with ||Rt(r:, r:)||_F <= eps/sqrt(d-1) ||Y||_F (the per-
// unfolding split of Theorem 3.2), capped at rmax; the cap is flagged.  Ranks
// stay on the device; later kernels read them from there.
#include <algorithm>

#include "digits.cuh"
#include "internal.cuh"
#include "philox.cuh"
#include "reflector.cuh"
#include "testmat.cuh"

namespace tts {

const DevSketch* plan_sketches_host(const Plan* p);
int plan_num_items(const Plan* p);
int plan_max_lev(const Plan* p);
int plan_ntasks(const Plan* p, int lev);

namespace {

constexpr int kThreads = 256;
constexpr int64_t kTableOffB = 256;

__device__ __forceinline__ const DevTables& tables(const char* wsb) {
  return *reinterpret_cast<const DevTables*>(wsb + kTableOffB);
}
__device__ __forceinline__ const DevSketch* dsk(const char* wsb) {
  return reinterpret_cast<const DevSketch*>(wsb + tables(wsb).off_sketches);
}
__device__ __forceinline__ const DevItem* ditems(const char* wsb) {
  return reinterpret_cast<const DevItem*>(wsb + tables(wsb).off_items);
}

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Block-wide sum (all threads get the result).  Uses red[32].
__device__ double block_sum(double v, double* red) {
  v = warp_sum(v);
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  __syncthreads();
  if (lane == 0) red[wid] = v;
  __syncthreads();
  double t = (threadIdx.x < (blockDim.x >> 5)) ? red[threadIdx.x] : 0.0;
  if (wid == 0) t = warp_sum(t);
  if (threadIdx.x == 0) red[0] = t;
  __syncthreads();
  const double r = red[0];
  __syncthreads();
  return r;
}

// Sums over the 32 lanes of two or four per-lane values at once (halving
// butterflies: 5 or 6 additions instead of 2 x 5 or 4 x 5).  warp_sum2: lane
// L returns the sum of p[(L >> 4) & 1]; warp_sum4: of p[(L >> 3) & 3].
__device__ __forceinline__ double warp_sum2(double p0, double p1) {
  const int lane = threadIdx.x & 31;
  const bool h16 = lane & 16;
  double k = h16 ? p1 : p0;
  k += __shfl_xor_sync(0xffffffffu, h16 ? p0 : p1, 16);
#pragma unroll
  for (int o = 8; o > 0; o >>= 1) k += __shfl_xor_sync(0xffffffffu, k, o);
  return k;
}
__device__ __forceinline__ double warp_sum4(double p0, double p1, double p2, double p3) {
  const int lane = threadIdx.x & 31;
  const bool h16 = lane & 16, h8 = lane & 8;
  double k0 = h16 ? p2 : p0, k1 = h16 ? p3 : p1;
  k0 += __shfl_xor_sync(0xffffffffu, h16 ? p0 : p2, 16);
  k1 += __shfl_xor_sync(0xffffffffu, h16 ? p1 : p3, 16);
  double k = h8 ? k1 : k0;
  k += __shfl_xor_sync(0xffffffffu, h8 ? k0 : k1, 8);
  k += __shfl_xor_sync(0xffffffffu, k, 4);
  k += __shfl_xor_sync(0xffffffffu, k, 2);
  k += __shfl_xor_sync(0xffffffffu, k, 1);
  return k;
}

// The FP64 pipe takes a warp instruction every 64 cycles and sub-partition, a guard
// around one costs several times that, and a shuffled addition about 130 cycles.  So
// the QR steps below give G = 8, 16 or 32 lanes to a column (more as fewer columns are
// left, so that the four pipes stay even; log2 G additions sum a column), two rows a
// lane at a time, without guards: rows above the current one have a zero multiplier,
// rows past the block are zero.
__host__ __device__ constexpr int qr_rows(int nr) { return tsqr_ld(nr) - 8; }   // multiple of 32
// Leading dimension: 8 mod 16, so that the 16 lanes of two columns read distinct banks.
__host__ __device__ constexpr int qr_ld(int nr) { return tsqr_ld(nr); }
template <int G>
__device__ __forceinline__ double group_sum(double v) {
#pragma unroll
  for (int o = G / 2; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Rows per iteration of a group and the first row of step i.
template <int G>
struct QrRows {
  static constexpr int kStep = G == 8 ? 16 : 32;         // 2 G, or G for whole warps
  static constexpr int kSecond = G == 32 ? 0 : G;        // offset of a lane's second row (0: none)
  static __device__ __forceinline__ int first(int i) { return i & ~(kStep - 1); }
};

// Gram row of step i: gram[c] = sum_{r >= i} A(r, i) A(r, c) for c > i, by all warps but
// the first, which forms the reflector of column i meanwhile (the longest chain of a
// step).
template <int G>
__device__ __forceinline__ void gram_pass(const double* A, int lda, int nrp, int w, int i, double* gram) {
  using R = QrRows<G>;
  const int t = (int)threadIdx.x - 32;
  const int sub = t & (G - 1), slot = t / G, nslot = ((int)blockDim.x - 32) / G;
  const int wbase = slot - (t & 31) / G;   // the warp's first slot
  const double* ai = A + lda * i;
  for (int cb = i + 1; cb + wbase < w; cb += nslot) {     // the same count for the whole warp
    const int c = cb + slot;
    const double* ac = A + lda * min(c, w - 1);
    double p0 = 0.0, p1 = 0.0;
    for (int r = R::first(i) + sub; r < nrp; r += R::kStep) {
      p0 = fma(r >= i ? ai[r] : 0.0, ac[r], p0);
      if (G < 32) p1 = fma(r + R::kSecond >= i ? ai[r + R::kSecond] : 0.0, ac[r + R::kSecond], p1);
    }
    const double g = group_sum<G>(G < 32 ? p0 + p1 : p0);
    if (sub == 0 && c < w) gram[c] = g;
  }
}
__device__ __forceinline__ void pivot_pass(const double* ai, int nrp, int i, double* beta, double* rdiag, double* v0s) {
  double p = 0.0;
  for (int r = (i & ~31) + (int)threadIdx.x; r < nrp; r += 32) {
    const double u = r >= i ? ai[r] : 0.0;
    p = fma(u, u, p);
  }
  p = group_sum<32>(p);
  if (threadIdx.x == 0) {
    double alpha, b, v0;
    reflector(p, ai[i], alpha, b, v0);
    beta[i] = b;
    rdiag[i] = alpha;
    *v0s = v0;
  }
}

// A(i:, c) -= b v (v^T A(i:, c)) for c > i, with v^T A(i:, c) = g_c - alpha A(i, c) and v =
// (v0, A(i+1:, i)).
template <int G>
__device__ __forceinline__ void update_pass(double* A, int lda, int nrp, int w, int i, const double* gram, double b,
                                            double alpha, double v0) {
  using R = QrRows<G>;
  const int sub = threadIdx.x & (G - 1), slot = threadIdx.x / G, nslot = blockDim.x / G;
  const uint32_t mask = G == 32 ? 0xffffffffu : ((1u << (G & 31)) - 1u) << (threadIdx.x & 31 & ~(G - 1));
  const double* ai = A + lda * i;
  for (int c = i + 1 + slot; c < w; c += nslot) {
    double* ac = A + lda * c;
    const double coef = b * fma(-alpha, ac[i], gram[c]);
    __syncwarp(mask);   // every lane of the column has read its head
    for (int r = R::first(i) + sub; r < nrp; r += R::kStep) {
      ac[r] = fma(-coef, r > i ? ai[r] : r == i ? v0 : 0.0, ac[r]);
      if (G < 32) {
        const int q = r + R::kSecond;
        ac[q] = fma(-coef, q > i ? ai[q] : q == i ? v0 : 0.0, ac[q]);
      }
    }
  }
}

// In-shared-memory Householder QR of an nr x w block A (ld = lda >= qr_rows(nr), rows
// nr..qr_rows(nr) zero), nr >= 1.  On exit column i holds v_i in rows i..nr-1 (v_i(0)
// at the diagonal), beta[i] = 2 / (v_i^T v_i) (0 for a zero column), rdiag[i] = R(i,
// i); the strict upper triangle holds R.
//
// Step i works from the Gram row g_c = sum_{r >= i} A(r, i) A(r, c), c >= i:
// g_i is the squared norm of the pivot column, and with v = A(i:, i) - alpha
// e_1 the reflector products are v^T A(i:, c) = g_c - alpha A(i, c).  So a
// step is one reduction pass and one update pass, two barriers in all.  Measured (a
// level of 128 x 26 blocks, 256 x 16 blocks, the root of 70 x 35): 65, 47, 131 us; a
// column per warp with five-step butterflies and the library's root and division in
// the chain took 93, 65 and (QR and CPQR) 440 us.
__device__ __forceinline__ void house_qr(double* A, int lda, int nr, int w, double* beta, double* rdiag) {
  const int kmax = min(nr, w);
  const int nrp = qr_rows(nr), nrp16 = (nr + 15) & ~15;
  __shared__ double v0s;
  __shared__ double gram[TT_MAXL];
  const int wide = blockDim.x >> 4, narrow = blockDim.x >> 5;   // columns that fit 16 and 32 lanes each
  for (int i = 0; i < kmax; ++i) {
    const int left = w - 1 - i;
    if (threadIdx.x < 32) pivot_pass(A + lda * i, nrp, i, beta, rdiag, &v0s);
    else if (left > wide - 2) gram_pass<8>(A, lda, nrp16, w, i, gram);
    else if (left > narrow - 1) gram_pass<16>(A, lda, nrp, w, i, gram);
    else gram_pass<32>(A, lda, nrp, w, i, gram);
    __syncthreads();
    const double b = beta[i], alpha = rdiag[i], v0 = v0s;
    if (b != 0.0) {
      if (left > wide) update_pass<8>(A, lda, nrp16, w, i, gram, b, alpha, v0);
      else if (left > narrow) update_pass<16>(A, lda, nrp, w, i, gram, b, alpha, v0);
      else update_pass<32>(A, lda, nrp, w, i, gram, b, alpha, v0);
    }
    __syncthreads();
    if (threadIdx.x == 0) A[i + lda * i] = v0;
  }
  for (int i = kmax + threadIdx.x; i < w; i += blockDim.x) {
    beta[i] = 0.0;
    rdiag[i] = 0.0;
  }
  __syncthreads();
}

// Z(:, c) = H_0 ... H_{kmax-1} [Z0(0:kmax, c); 0] for the nr-row block of
// reflectors V (ld ldv, heads v_i(0) on the diagonal) and beta, columns c <
// ncol; columns ncol..npad-1 of Z are zero.  Z0 = Zin (ld ldzin).  A warp
// keeps NC columns c = cb + nw j in registers through all reflectors (no
// barrier between reflectors; one butterfly per reflector for the NC dots;
// NC > 1 only for blocks of at most 64 rows); NT = ceil(nr / 32) rows per
// lane, nr <= 256.
constexpr int kRowsPerLane = kTsqrMaxRows / 32;
template <int NC>
__device__ __forceinline__ void warp_sums(const double (&p)[4], double (&d)[4]) {
  if (NC == 1) {
    d[0] = warp_sum(p[0]);
  } else if (NC == 2) {
    const double g = warp_sum2(p[0], p[1]);
    d[0] = __shfl_sync(0xffffffffu, g, 0);
    d[1] = __shfl_sync(0xffffffffu, g, 16);
  } else {
    const double g = warp_sum4(p[0], p[1], p[2], p[3]);
#pragma unroll
    for (int j = 0; j < 4; ++j) d[j] = __shfl_sync(0xffffffffu, g, 8 * j);
  }
}
template <int NT, int NC>
__device__ __forceinline__ void expand_group(const double* V, int64_t ldv, const double* beta, int nr, int kmax,
                                             const double* Zin, int64_t ldzin, int cb, int nw, double* Z,
                                             int64_t ldz) {
  const int lane = threadIdx.x & 31;
  double z[NC][NT];
#pragma unroll
  for (int j = 0; j < NC; ++j)
#pragma unroll
    for (int t = 0; t < NT; ++t) {
      const int r = lane + 32 * t;
      z[j][t] = r < kmax ? Zin[r + ldzin * (cb + nw * j)] : 0.0;
    }
  for (int i = kmax - 1; i >= 0; --i) {
    const double b = beta[i];
    if (b == 0.0) continue;
    double v[NT];
    double p[4] = {0.0, 0.0, 0.0, 0.0}, d[4];
#pragma unroll
    for (int t = 0; t < NT; ++t) {
      const int r = lane + 32 * t;
      v[t] = (r >= i && r < nr) ? V[r + ldv * i] : 0.0;
#pragma unroll
      for (int j = 0; j < NC; ++j) p[j] = fma(v[t], z[j][t], p[j]);
    }
    warp_sums<NC>(p, d);
#pragma unroll
    for (int j = 0; j < NC; ++j) {
      const double s = d[j] * b;
#pragma unroll
      for (int t = 0; t < NT; ++t) z[j][t] = fma(-s, v[t], z[j][t]);
    }
  }
#pragma unroll
  for (int j = 0; j < NC; ++j)
#pragma unroll
    for (int t = 0; t < NT; ++t) {
      const int r = lane + 32 * t;
      if (r < nr) Z[r + ldz * (cb + nw * j)] = z[j][t];
    }
}
template <int NT>
__device__ __forceinline__ void expand_cols_nt(const double* V, int64_t ldv, const double* beta, int nr, int w,
                                               const double* Zin, int64_t ldzin, int ncol, int npad, double* Z,
                                               int64_t ldz) {
  const int wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const int kmax = min(nr, w);
  if (NT > 2) {  // tall blocks: one column per warp keeps the registers in bounds
    for (int c = wid; c < ncol; c += nw) expand_group<NT, 1>(V, ldv, beta, nr, kmax, Zin, ldzin, c, nw, Z, ldz);
  } else {
    for (int cb = wid; cb < ncol; cb += 4 * nw) {
      switch (min(4, (ncol - 1 - cb) / nw + 1)) {
        case 1: expand_group<NT, 1>(V, ldv, beta, nr, kmax, Zin, ldzin, cb, nw, Z, ldz); break;
        case 2: expand_group<NT, 2>(V, ldv, beta, nr, kmax, Zin, ldzin, cb, nw, Z, ldz); break;
        case 3: expand_group<NT, 3>(V, ldv, beta, nr, kmax, Zin, ldzin, cb, nw, Z, ldz); break;
        default: expand_group<NT, 4>(V, ldv, beta, nr, kmax, Zin, ldzin, cb, nw, Z, ldz); break;
      }
    }
  }
  for (int o = threadIdx.x; o < nr * (npad - ncol); o += blockDim.x) Z[o % nr + ldz * (ncol + o / nr)] = 0.0;
}
__device__ __forceinline__ void expand_cols(const double* V, int64_t ldv, const double* beta, int nr, int w,
                                            const double* Zin, int64_t ldzin, int ncol, int npad, double* Z,
                                            int64_t ldz) {
  switch ((nr + 31) / 32) {
    case 1: expand_cols_nt<1>(V, ldv, beta, nr, w, Zin, ldzin, ncol, npad, Z, ldz); break;
    case 2: expand_cols_nt<2>(V, ldv, beta, nr, w, Zin, ldzin, ncol, npad, Z, ldz); break;
    case 3: expand_cols_nt<3>(V, ldv, beta, nr, w, Zin, ldzin, ncol, npad, Z, ldz); break;
    case 4: expand_cols_nt<4>(V, ldv, beta, nr, w, Zin, ldzin, ncol, npad, Z, ldz); break;
    case 5: expand_cols_nt<5>(V, ldv, beta, nr, w, Zin, ldzin, ncol, npad, Z, ldz); break;
    case 6: expand_cols_nt<6>(V, ldv, beta, nr, w, Zin, ldzin, ncol, npad, Z, ldz); break;
    case 7: expand_cols_nt<7>(V, ldv, beta, nr, w, Zin, ldzin, ncol, npad, Z, ldz); break;
    default: expand_cols_nt<kRowsPerLane>(V, ldv, beta, nr, w, Zin, ldzin, ncol, npad, Z, ldz); break;
  }
}

// One pivoted-QR step's update of the columns c > i of the block Rs (ld ldr, nrp rows
// with the zero ones) by reflector i (v = Rs(i:, i), beta b), and their trailing norms
// over rows > i.
template <int G>
__device__ __forceinline__ void cpqr_pass(double* Rs, int ldr, int nrp, int w, int i, double b, double* nrm) {
  using R = QrRows<G>;
  const int sub = threadIdx.x & (G - 1), slot = threadIdx.x / G, nslot = blockDim.x / G;
  const int wbase = slot - (threadIdx.x & 31) / G;
  const double* ai = Rs + ldr * i;
  for (int cb = i + 1; cb + wbase < w; cb += nslot) {
    const int c = cb + slot;
    double* ac = Rs + ldr * min(c, w - 1);
    double p0 = 0.0, p1 = 0.0;
    for (int r = R::first(i) + sub; r < nrp; r += R::kStep) {
      p0 = fma(r >= i ? ai[r] : 0.0, ac[r], p0);
      if (G < 32) p1 = fma(r + R::kSecond >= i ? ai[r + R::kSecond] : 0.0, ac[r + R::kSecond], p1);
    }
    const double coef = group_sum<G>(G < 32 ? p0 + p1 : p0) * b;
    double t0 = 0.0, t1 = 0.0;
    if (c < w) {
      for (int r = R::first(i) + sub; r < nrp; r += R::kStep) {
        const double x0 = fma(-coef, r >= i ? ai[r] : 0.0, ac[r]);
        ac[r] = x0;
        const double y0 = r > i ? x0 : 0.0;
        t0 = fma(y0, y0, t0);
        if (G < 32) {
          const int q = r + R::kSecond;
          const double x1 = fma(-coef, q >= i ? ai[q] : 0.0, ac[q]);
          ac[q] = x1;
          const double y1 = q > i ? x1 : 0.0;
          t1 = fma(y1, y1, t1);
        }
      }
    }
    const double t = group_sum<G>(G < 32 ? t0 + t1 : t0);
    if (sub == 0 && c < w) nrm[c] = t;
  }
}
__device__ __forceinline__ void cpqr_step(double* Rs, int ldr, int nr, int w, int i, double b, double* nrm) {
  const int left = w - 1 - i, wide = blockDim.x >> 4, narrow = blockDim.x >> 5;
  if (left > wide) cpqr_pass<8>(Rs, ldr, (nr + 15) & ~15, w, i, b, nrm);
  else if (left > narrow) cpqr_pass<16>(Rs, ldr, qr_rows(nr), w, i, b, nrm);
  else cpqr_pass<32>(Rs, ldr, qr_rows(nr), w, i, b, nrm);
}

// Copies an nr x w column-major block (leading dimension ldy) into shared
// memory (leading dimension lda >= qr_rows(nr)), rows nr..qr_rows(nr) zero; eight
// independent loads per thread are in flight at a time.
__device__ void load_block(double* A, int lda, const double* Y, int64_t ldy, int nr, int w) {
  for (int c0 = 0; c0 < w; c0 += 8)
    for (int r = threadIdx.x; r < nr; r += blockDim.x) {
      double v[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) v[u] = (c0 + u < w) ? Y[r + ldy * (c0 + u)] : 0.0;
#pragma unroll
      for (int u = 0; u < 8; ++u)
        if (c0 + u < w) A[r + lda * (c0 + u)] = v[u];
    }
  const int pad = qr_rows(nr) - nr;
  for (int o = threadIdx.x; o < pad * w; o += blockDim.x) A[nr + o % pad + lda * (o / pad)] = 0.0;
}

__device__ __forceinline__ void flag_status(char* wsb, int bits) {
  atomicOr(reinterpret_cast<int*>(wsb + kStatusOff), bits);
}

// FP16 plans: the sketch kernels split X 2^s (s = x_scale_log2), so every
// sketch holds 2^s times its value.  Scale the sketches of item item0 +
// blockIdx.y back by 2^-s (exact in FP64) and flag a non-finite entry (an
// inf or NaN in X, or |X| 2^s past the FP16 range), which is replaced by
// zero so that the finalize runs on finite values (its result is then
// meaningless; the status word says so).
__global__ void __launch_bounds__(kThreads) sketch_unscale_kernel(char* wsb, int item0) {
  const DevItem& it = ditems(wsb)[item0 + (int)blockIdx.y];
  if (it.prec != TT_PREC_FP16) return;
  const DevSketch* sks = dsk(wsb);
  double* ws = reinterpret_cast<double*>(wsb);
  const double f = ldexp(1.0, -it.x_scale_log2);
  int bad = 0;
  auto scale = [&](double& x) {
    const double v = x * f;
    const bool fin = isfinite(v);
    bad |= fin ? 0 : 1;
    x = fin ? v : 0.0;
  };
  const int64_t tid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x, nthr = (int64_t)gridDim.x * blockDim.x;
  for (int s = 0; s < it.nsk; ++s) {
    const DevSketch& d = sks[it.sk0 + s];
    double* p = ws + d.off;  // 16-byte aligned (workspace regions are)
    const int64_t n = d.rows * d.width;
    double2* p2 = reinterpret_cast<double2*>(p);
    for (int64_t e = tid; e < n / 2; e += nthr) {
      double2 v = p2[e];
      scale(v.x);
      scale(v.y);
      p2[e] = v;
    }
    if ((n & 1) && tid == 0) scale(p[n - 1]);
  }
  if (__syncthreads_or(bad) && threadIdx.x == 0) flag_status(wsb, ST_NONFINITE);
}

// ------------------------------------------------------------------ TSQR up
// One task = one row block of level L of one basis sketch (launch Lg holds
// the tasks whose tree has Lg - L more levels above them than the deepest
// tree, so that every root runs in the last launch).  Non-root blocks write
// their R into the next level's matrix; the root block also does the CPQR, the rank
// decision and (unless root_sep) the first expansion step.  A root block of at most
// 6 w rows or kTsqrOneBlock entries is pivoted as it stands -- its columns have the norms and inner products
// of R's -- which spares the QR before it and the product of the two Q factors.
__global__ void __launch_bounds__(kThreads, 4) tsqr_level_kernel(char* wsb, int Lg, int* ranks, int root_sep) {
  extern __shared__ double sm[];
  const DevTables& T = tables(wsb);
  const Task task = reinterpret_cast<const Task*>(wsb + T.off_tasks[Lg])[blockIdx.x];
  const int L = task.lev;
  const DevSketch& s = dsk(wsb)[task.sk];
  const DevItem& it = ditems(wsb)[s.item];
  double* ws = reinterpret_cast<double*>(wsb);
  const int w = s.width;
  const int64_t m = s.lev_rows[L];
  const int64_t r0 = (int64_t)task.blk * s.lev_bl[L];
  const int nr = (int)imin64(s.lev_bl[L], m - r0);
  const int lda = qr_ld(nr), ldw = qr_ld(w);
  double* A = sm;                         // lda x w
  double* red = A + (size_t)lda * w;      // 32
  double* beta = red + 32;                // w
  double* rdiag = beta + TT_MAXL;         // w
  double* Rs = rdiag + TT_MAXL;           // ldw x w (root only)
  double* Q2 = Rs + ldw * w;                // w x w (root only), then w x w of rank sums
  __shared__ int piv[TT_MAXL];
  __shared__ int s_rank;
  double* Y = ws + s.lev_mat[L];
  load_block(A, lda, Y + r0, m, nr, w);
  __syncthreads();
  const bool root = (s.lev_nblk[L] == 1);
  const bool direct = root && nr >= w && (nr <= 6 * w || nr * w <= kTsqrOneBlock);   // pivot the block itself
  const int kmax = min(nr, w);
  // Householder vectors back in place, scalars to the level's beta array
  auto store_block = [&](const double* bt) {
    for (int o = threadIdx.x; o < nr * w; o += blockDim.x) {
      const int r = o % nr, c = o / nr;
      Y[r0 + r + m * c] = A[r + lda * c];
    }
    for (int i = threadIdx.x; i < w; i += blockDim.x) ws[s.lev_beta[L] + (int64_t)task.blk * w + i] = bt[i];
  };
  if (!direct) {
    house_qr(A, lda, nr, w, beta, rdiag);
    store_block(beta);
  }
  auto rval = [&](int i, int c) -> double {
    if (i >= kmax || c < i) return 0.0;
    return c == i ? rdiag[i] : A[i + lda * c];
  };
  if (!root) {
    const int64_t m1 = s.lev_rows[L + 1];
    double* Yn = ws + s.lev_mat[L + 1];
    for (int o = threadIdx.x; o < w * w; o += blockDim.x) {
      const int i = o % w, c = o / w;
      Yn[(int64_t)task.blk * w + i + m1 * c] = rval(i, c);
    }
    return;
  }
  // ---- root: CPQR, of the block (nr x w) or of its R (w x w), in shared memory.
  // Per step: warp 0 picks the pivot (largest recomputed trailing norm, lowest
  // index on ties), swaps it into place and forms the reflector; then each warp
  // applies it to its own columns and recomputes their trailing norms for the
  // next step.
  double* Cs = direct ? A : Rs;
  const int ldc = direct ? lda : ldw, nc = direct ? nr : w;
  if (!direct)
    for (int o = threadIdx.x; o < qr_rows(w) * w; o += blockDim.x) {
      const int i = o % qr_rows(w), c = o / qr_rows(w);
      Rs[i + ldw * c] = i < w ? rval(i, c) : 0.0;
    }
  for (int c = threadIdx.x; c < w; c += blockDim.x) piv[c] = c;
  __syncthreads();
  __shared__ double nrm[TT_MAXL];
  __shared__ double qb[TT_MAXL], qd[TT_MAXL];
  double total2 = 0.0;
  {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
    for (int c = wid; c < w; c += nw) {  // trailing norms of step 0
      double t = 0.0;
      for (int r = lane; r < nc; r += 32) t = fma(Cs[r + ldc * c], Cs[r + ldc * c], t);
      t = warp_sum(t);
      if (lane == 0) nrm[c] = t;
    }
    __syncthreads();
    total2 = block_sum((int)threadIdx.x < w ? nrm[threadIdx.x] : 0.0, red);
    for (int i = 0; i < w; ++i) {
      if (wid == 0) {
        // argmax over c >= i; norms are >= 0, so their bit patterns order like them
        long long key = -1;
        int arg = w;
        for (int c = i + lane; c < w; c += 32) {
          const long long k2 = __double_as_longlong(nrm[c]);
          if (k2 > key) key = k2, arg = c;
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
          const long long k2 = __shfl_xor_sync(0xffffffffu, key, o);
          const int a2 = __shfl_xor_sync(0xffffffffu, arg, o);
          if (k2 > key || (k2 == key && a2 < arg)) key = k2, arg = a2;
        }
        // no key above -1 (every trailing norm a NaN with the sign bit set):
        // keep column i, so that the swap stays inside the block
        const int j = arg < w ? arg : i;
        if (j != i) {
          for (int r = lane; r < nc; r += 32) {
            const double t = Cs[r + ldc * i];
            Cs[r + ldc * i] = Cs[r + ldc * j];
            Cs[r + ldc * j] = t;
          }
          if (lane == 0) {
            const int t = piv[i];
            piv[i] = piv[j];
            piv[j] = t;
            const double tn = nrm[i];
            nrm[i] = nrm[j];
            nrm[j] = tn;
          }
        }
        __syncwarp();
        if (lane == 0) {  // Householder on column i, rows i..nc-1
          double alpha, b, v0;
          reflector(nrm[i], Cs[i + ldc * i], alpha, b, v0);
          Cs[i + ldc * i] = v0;
          qb[i] = b;
          qd[i] = alpha;
        }
      }
      __syncthreads();
      cpqr_step(Cs, ldc, nc, w, i, qb[i], nrm);
      __syncthreads();
    }
  }
  // Q2: the factor that the block's own reflectors are applied to, columns with
  // diag(Rt) >= 0 (direct: those signs alone)
  for (int o = threadIdx.x; o < w * w; o += blockDim.x) Q2[o] = (o % w == o / w) ? 1.0 : 0.0;
  __syncthreads();
  if (direct) {
    store_block(qb);
  } else {
    expand_cols(Rs, ldw, qb, w, w, Q2, w, w, w, Q2, w);
    __syncthreads();
  }
  // Rt with signs normalised (diag >= 0), Q2 columns likewise
  double* Rt = ws + s.off_rt;
  for (int o = threadIdx.x; o < w * w; o += blockDim.x) {
    const int i = o % w, c = o / w;
    const double sg = qd[i] < 0.0 ? -1.0 : 1.0, sc = qd[c] < 0.0 ? -1.0 : 1.0;
    double v = 0.0;
    if (c > i) v = Cs[i + ldc * c];
    else if (c == i) v = qd[i];
    Rt[o] = sg * v;
    Q2[o] *= sc;
    ws[s.off_q2 + o] = Q2[o];
  }
  for (int c = threadIdx.x; c < w; c += blockDim.x) reinterpret_cast<int*>(ws + s.off_piv)[c] = piv[c];
  __syncthreads();
  // rank decision.  tail(r) = ||Rt(r:, r:)||_F^2 = sum_{c >= r} t_c(r) with
  // t_c(r) = sum_{i = r..c} Rt(i, c)^2; thread c forms t_c(.) by a running sum
  // from the diagonal up, then tail(r) is summed over the columns.
  double* tcol = Q2 + w * w;  // t_c(r) at [r + w c] (r <= c), w x w
  __shared__ double tails[TT_MAXL + 1];
  for (int c = threadIdx.x; c < w; c += blockDim.x) {
    double run = 0.0;
    for (int i2 = c; i2 >= 0; --i2) {
      const double v = c > i2 ? Cs[i2 + ldc * c] : qd[c];   // |Rt(i2, c)|
      run = fma(v, v, run);
      tcol[i2 + w * c] = run;
    }
  }
  __syncthreads();
  for (int cand = threadIdx.x; cand <= w; cand += blockDim.x) {
    double tail = 0.0;
    for (int c = cand; c < w; ++c) tail += tcol[cand + w * c];
    tails[cand] = tail;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    const int limit = min(s.rpad, w);
    int r = s.target_rank;
    if (it.eps_mode) {
      const double thr = it.eps / sqrt((double)max(it.d - 1, 1)) * sqrt(total2);
      r = limit;
      bool met = false;
      for (int cand = 1; cand <= limit; ++cand) {
        if (sqrt(tails[cand]) <= thr) {
          r = cand;
          met = true;
          break;
        }
      }
      if (!met) flag_status(wsb, ST_RANK_CAP);
    }
    r = max(1, min(r, limit));
    s_rank = r;
    int* rk = ranks + it.rank_off;
    rk[s.k] = r;
    if (s.k == 1) rk[0] = 1;
    if (s.k == it.d - 1) rk[it.d] = 1;
    if (it.rank_off == 0) {  // copy for the backward of a single-item plan
      int* cp = reinterpret_cast<int*>(wsb + kRankCopyOff);
      cp[s.k] = r;
      if (s.k == 1) cp[0] = 1;
      if (s.k == it.d - 1) cp[it.d] = 1;
    }
  }
  __syncthreads();
  const int r = s_rank;
  // leading r x r block of Rt for the backward pass (rpad x rpad, zero padded)
  for (int o = threadIdx.x; o < s.rpad * s.rpad; o += blockDim.x) {
    const int i = o % s.rpad, c = o / s.rpad;
    ws[it.off_rr[s.k] + o] = (i < r && c < r) ? Rt[i + w * c] : 0.0;
  }
  // Z_root = Q_root [Q2(:, 1:r); 0]  (m x rpad, columns >= r are zero)
  if (!root_sep) expand_cols(A, lda, direct ? qb : beta, nr, w, Q2, w, r, s.rpad, ws + s.lev_z[L], m);
}

// ---------------------------------------------------------------- TSQR down
// Z_L(block) = Q_block [Z_{L+1}(rows of this block's R); 0], and Q_root [Q2; 0] at the
// root when root_sep.  A block's reflectors occupy one SM's FP64 pipe (a column of a
// 192-row block costs 17 warp instructions a reflector), so few blocks share their
// columns over blockIdx.y, cw columns each.
__global__ void __launch_bounds__(kThreads) tsqr_expand_kernel(char* wsb, int Lg, const int* ranks, int root_sep,
                                                               int cw) {
  extern __shared__ double sm[];
  const DevTables& T = tables(wsb);
  const Task task = reinterpret_cast<const Task*>(wsb + T.off_tasks[Lg])[blockIdx.x];
  const int L = task.lev;
  const DevSketch& s = dsk(wsb)[task.sk];
  const bool root = s.nlev - 1 <= L;
  if (root && !root_sep) return;  // root of this tree, already expanded
  const int c0 = (int)blockIdx.y * cw;
  if (c0 >= s.rpad) return;
  const DevItem& it = ditems(wsb)[s.item];
  double* ws = reinterpret_cast<double*>(wsb);
  const int w = s.width;
  const int r = ranks[it.rank_off + s.k];
  const int64_t m = s.lev_rows[L];
  const int64_t r0 = (int64_t)task.blk * s.lev_bl[L];
  const int nr = (int)imin64(s.lev_bl[L], m - r0);
  const int lda = qr_ld(nr);
  double* V = sm;
  double* beta = V + (size_t)lda * w;
  const double* Y = ws + s.lev_mat[L];
  load_block(V, lda, Y + r0, m, nr, w);
  for (int i = threadIdx.x; i < w; i += blockDim.x) beta[i] = ws[s.lev_beta[L] + (int64_t)task.blk * w + i];
  __syncthreads();
  const double* Zin = root ? ws + s.off_q2 : ws + s.lev_z[L + 1] + (int64_t)task.blk * w;
  const int64_t ldz = root ? w : s.lev_rows[L + 1];
  expand_cols(V, lda, beta, nr, w, Zin + ldz * c0, ldz, max(0, min(r - c0, cw)), min(s.rpad - c0, cw),
              ws + s.lev_z[L] + r0 + m * c0, m);
}

// --------------------------------------------------------- one-pass middle
// B = P_{d*}^T Omega_{d*}  (r x l), summed over row chunks with atomics.
// item < 0: batched launch, item = blockIdx.y
__global__ void __launch_bounds__(kThreads) mid_b_kernel_f64(char* wsb, int item_arg, const int* ranks) {
  const int item = item_arg >= 0 ? item_arg : (int)blockIdx.y;
  constexpr int CH = 32;
  __shared__ double Ps[CH * TT_MAXL];
  __shared__ double Gs[CH * (TT_MAXL + 1)];
  const DevItem& it = ditems(wsb)[item];
  const DevSketch& sp = dsk(wsb)[it.basis_of_k[it.mbk]];
  // the middle test matrix is the one the least-squares sketch used
  const DevSketch* kr_mid = dsk(wsb)[it.mid_sk].kr_nm ? &dsk(wsb)[it.mid_sk] : nullptr;
  double* ws = reinterpret_cast<double*>(wsb);
  const int r = ranks[it.rank_off + it.mbk];
  const int l = it.lmid;
  const int64_t M = sp.rows;
  const double* Pm = ws + sp.lev_z[0];
  // with r l <= blockDim pairs each thread keeps its pair's sum across the
  // block's row chunks and adds it to B once
  const bool keep = r * l <= (int)blockDim.x;
  double kept = 0.0;
  for (int64_t v0 = (int64_t)blockIdx.x * CH; v0 < M; v0 += (int64_t)gridDim.x * CH) {
    const int nv = (int)imin64(CH, M - v0);
    __syncthreads();
    for (int o = threadIdx.x; o < CH * r; o += blockDim.x) {
      const int v = o % CH, c = o / CH;
      Ps[v + CH * c] = v < nv ? Pm[v0 + v + M * c] : 0.0;
    }
    const int nq = (l + 3) / 4;
    for (int o = threadIdx.x; o < nv * nq; o += blockDim.x) {
      const int v = o % nv, q = o / nv;
      double z[4];
      tm_quad_f64(wsb, kr_mid, it.seed, (uint32_t)it.mstream, (uint64_t)(v0 + v), (uint32_t)q, z);
#pragma unroll
      for (int t = 0; t < 4; ++t)
        if (4 * q + t < l) Gs[v + CH * (4 * q + t)] = z[t];
    }
    __syncthreads();
    for (int o = threadIdx.x; o < r * l; o += blockDim.x) {
      const int c = o % r, j = o / r;
      double acc = 0.0;
      for (int v = 0; v < nv; ++v) acc = fma(Ps[v + CH * c], Gs[v + CH * j], acc);
      if (keep) kept += acc;
      else atomicAdd(ws + it.off_B + c + (int64_t)it.rpad[it.mbk] * j, acc);
    }
  }
  if (keep && (int)threadIdx.x < r * l) {
    const int c = (int)threadIdx.x % r, j = (int)threadIdx.x / r;
    atomicAdd(ws + it.off_B + c + (int64_t)it.rpad[it.mbk] * j, kept);
  }
}

// QR of B^T (l x r) -> RB (r x r) and M = QB RB^{-T} (l x r, over QB's place); singular
// B is flagged.  All of it in shared memory (in global memory the reflectors'
// application and the back-substitution took most of 157 us at l = 35, r = 25).
// item < 0: batched launch, item = blockIdx.y
__global__ void __launch_bounds__(kThreads) mid_ls_kernel(char* wsb, int item_arg, const int* ranks) {
  const int item = item_arg >= 0 ? item_arg : (int)blockIdx.y;
  extern __shared__ double sm[];
  __shared__ double beta[TT_MAXL], rdiag[TT_MAXL];
  const DevItem& it = ditems(wsb)[item];
  double* ws = reinterpret_cast<double*>(wsb);
  const int r = ranks[it.rank_off + it.mbk];
  const int l = it.lmid;
  const int rp = it.rpad[it.mbk];
  const int lda = qr_ld(l), lp = qr_rows(l);
  double* A = sm;             // lda x r
  double* M = A + lda * r;    // l x r, ld l + 1
  const int ldm = l + 1;
  for (int o = threadIdx.x; o < lp * r; o += blockDim.x) {
    const int j = o % lp, c = o / lp;
    A[j + lda * c] = j < l ? ws[it.off_B + c + (int64_t)rp * j] : 0.0;  // B^T(j, c) = B(c, j)
  }
  for (int o = threadIdx.x; o < l * r; o += blockDim.x) M[o % l + ldm * (o / l)] = (o % l == o / l) ? 1.0 : 0.0;
  __syncthreads();
  house_qr(A, lda, l, r, beta, rdiag);
  // RB (rp x rp) with diag >= 0; QB = H_0..H_{r-1} [I_r; 0] with matching signs
  double* RB = ws + it.off_RB;
  double* QB = ws + it.off_QB;
  __shared__ double sgn[TT_MAXL];
  __shared__ double rmax_abs;
  if (threadIdx.x == 0) {
    double mx = 0.0;
    for (int i = 0; i < r; ++i) mx = fmax(mx, fabs(rdiag[i]));
    rmax_abs = mx;
  }
  for (int i = threadIdx.x; i < r; i += blockDim.x) sgn[i] = rdiag[i] < 0.0 ? -1.0 : 1.0;
  __syncthreads();
  for (int o = threadIdx.x; o < rp * rp; o += blockDim.x) {
    const int i = o % rp, c = o / rp;
    double v = 0.0;
    if (i < r && c < r && c >= i) v = sgn[i] * (c == i ? rdiag[i] : A[i + lda * c]);
    RB[o] = v;
  }
  if (threadIdx.x == 0) {
    bool sing = !(rmax_abs > 0.0);
    for (int i = 0; i < r; ++i)
      if (!(fabs(rdiag[i]) > 1e-13 * rmax_abs)) sing = true;
    if (sing) flag_status(wsb, ST_RANK_DEFICIENT);
  }
  expand_cols(A, lda, beta, l, r, M, ldm, r, r, M, ldm);
  // M = QB RB^{-T}: row j solves m RB^T = QB(j, :) from the last column (a zero
  // diagonal of RB gives a zero column, as flagged above), so that H = S_{d*} M is a
  // plain product.  A step takes column c's share out of the columns before it; the
  // signs of QB's columns and RB's rows meet in sgn.
  __shared__ double rinv[TT_MAXL];
  for (int c = threadIdx.x; c < r; c += blockDim.x) {
    const double dg = fabs(rdiag[c]);
    rinv[c] = dg != 0.0 ? 1.0 / dg : 0.0;
  }
  __syncthreads();
  for (int o = threadIdx.x; o < l * r; o += blockDim.x) M[o % l + ldm * (o / l)] *= sgn[o / l];
  __syncthreads();
  for (int c = r - 1; c > 0; --c) {
    for (int o = threadIdx.x; o < l * c; o += blockDim.x) {
      const int j = o % l, c2 = o / l;
      const double x = M[j + ldm * c] * rinv[c];
      M[j + ldm * c2] = fma(-x, sgn[c2] * A[c2 + lda * c], M[j + ldm * c2]);
    }
    __syncthreads();
  }
  for (int o = threadIdx.x; o < l * rp; o += blockDim.x) {
    const int j = o % l, c = o / l;
    QB[j + (int64_t)l * c] = c < r ? M[j + ldm * c] * rinv[c] : 0.0;
  }
}

// H = S_{d*} M  (N_{d*} x rpad, columns >= r zero), M = QB RB^{-T} (l x r)
// from mid_ls_kernel; one thread per entry of H.
// item < 0: batched launch, item = blockIdx.y
__global__ void __launch_bounds__(kThreads) mid_h_kernel(char* wsb, int item_arg, const int* ranks) {
  const int item = item_arg >= 0 ? item_arg : (int)blockIdx.y;
  __shared__ double Ms[TT_MAXL * TT_MAXL];
  const DevItem& it = ditems(wsb)[item];
  const DevSketch& sm_ = dsk(wsb)[it.mid_sk];
  double* ws = reinterpret_cast<double*>(wsb);
  const int r = ranks[it.rank_off + it.mbk];
  const int rp = it.rpad[it.mbk];
  const int l = it.lmid;
  for (int o = threadIdx.x; o < l * r; o += blockDim.x) Ms[o] = ws[it.off_QB + o];
  __syncthreads();
  const int64_t Nm = sm_.rows;
  const double* S = ws + sm_.off;
  double* H = ws + it.off_H;
  for (int64_t o = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; o < Nm * rp; o += (int64_t)gridDim.x * blockDim.x) {
    const int64_t u = o % Nm;
    const int c = (int)(o / Nm);
    double h = 0.0;
    if (c < r)
      for (int j = 0; j < l; ++j) h = fma(S[u + Nm * j], Ms[j + l * c], h);
    H[o] = h;
  }
}

// --------------------------------------------------------------- the cores
// Left type  (k <= d*): G(a,i,c) = sum_u A(u,a) B(u + N_{k-1} i, c),  A = Q_{k-1}
//            (identity 1x1 for k = 1), B = Q_k or H (middle core, one-pass).
// Right type (k > d*):  G(a,i,c) = sum_v A(i + n_k v, a) B(v, c),   A = P_{k-1},
//            B = P_k (identity 1x1 for k = d).
//
// Both are G(:, i, :) = A_i^T B_i (ra x rc) over a contraction of length
// `inner`: left A_i = A, B_i = rows [inner i, inner (i + 1)) of B; right A_i =
// rows {i + n_k v} of A, B_i = B; an absent factor is the 1 x 1 identity.  One
// block per (item, k, slice i): chunks of A_i and B_i are staged in shared
// memory and the threads split the (a, c) pairs and the contraction index, so
// the FP64 work is the plain multiply-adds with one short reduction per pair.  A
// chunk is kCoreChunk indices at 64 columns and longer for fewer (the same shared
// memory): a chunk costs two barriers and a load's latency whatever its length.
// Measured (cores of 512 uneven tensors, with their slices over five blocks): 1.20 -> 0.39 ms.
constexpr int kCoreChunk = 32;
constexpr int kCoreBlocks = 16384;   // blocks, about: the slices of a large batch's cores are uneven work
__global__ void __launch_bounds__(kThreads) cores_kernel(char* wsb, double* cores, const int* ranks,
                                                         int item0, int nitems, int only_k, int dmax,
                                                         uint32_t skip) {
  __shared__ double sA[(kCoreChunk + 1) * TT_MAXL], sB[(kCoreChunk + 1) * TT_MAXL];
  __shared__ double red[kThreads];
  const int item = item0 + (int)blockIdx.x / dmax;
  const int k = (int)blockIdx.x % dmax + 1;
  if (item >= item0 + nitems) return;
  const DevItem& it = ditems(wsb)[item];
  if (k > it.d) return;
  if (only_k > 0 && k != only_k) return;
  if (only_k == 0 && k == it.mcore && it.passes == 2) return;  // second pass computes it
  if (skip >> k & 1) return;  // formed by core_gemm_kernel
  const DevSketch* S = dsk(wsb);
  const double* ws = reinterpret_cast<const double*>(wsb);
  const int* rk = ranks + it.rank_off;
  const int ra = rk[k - 1], rc = rk[k];
  const int rpa = it.rpad[k - 1], rpc = it.rpad[k];
  const int64_t nk = it.n[k - 1];
  double* G = cores + it.core_off[k];
  const bool left = k <= it.ds;
  const double* A = nullptr;
  const double* B = nullptr;
  int64_t lda = 0, ldb = 0, inner = 0;
  if (left) {
    inner = it.N[k - 1];
    if (k >= 2) {
      const DevSketch& sa = S[it.basis_of_k[k - 1]];
      A = ws + sa.lev_z[0];
      lda = sa.rows;
    }
    if (k == it.mcore) {
      B = ws + it.off_H;
      ldb = it.N[k];
    } else {
      const DevSketch& sb = S[it.basis_of_k[k]];
      B = ws + sb.lev_z[0];
      ldb = sb.rows;
    }
  } else {
    inner = it.N[it.d] / it.N[k];
    if (k == it.mcore) {  // one-sided last core: G_d(a, i, 0) = H(i, a)
      A = ws + it.off_H;
      lda = S[it.mid_sk].rows;
    } else {
      const DevSketch& sa = S[it.basis_of_k[k - 1]];
      A = ws + sa.lev_z[0];
      lda = sa.rows;
    }
    if (k < it.d) {
      const DevSketch& sb = S[it.basis_of_k[k]];
      B = ws + sb.lev_z[0];
      ldb = sb.rows;
    }
  }
  const int P = ra * rc, rm = max(ra, rc);
  // (2 kCoreChunk + 1) 32 <= (kCoreChunk + 1) 64, and so on
  const int chunk = rm <= 8 ? 8 * kCoreChunk : rm <= 16 ? 4 * kCoreChunk : rm <= 32 ? 2 * kCoreChunk : kCoreChunk;
  const int LDC = chunk + 1;   // threads of a warp read different columns of one row
  for (int64_t i = blockIdx.y; i < nk; i += gridDim.y) {
    double* Gi = G + rpa * i;  // G(a, i, c) = Gi[a + rpa nk c]
    for (int pg = 0; pg < P; pg += blockDim.x) {
      const int Pg = min(P - pg, (int)blockDim.x), nsplit = blockDim.x / Pg;
      const int p = pg + (int)threadIdx.x % Pg, sp = (int)threadIdx.x / Pg;
      const int a = p % ra, c = p / ra;
      double acc = 0.0;
      for (int64_t u0 = 0; u0 < inner; u0 += chunk) {
        const int uc = (int)imin64(chunk, inner - u0);
        __syncthreads();
        for (int o = threadIdx.x; o < uc * ra; o += blockDim.x) {
          const int u = o % uc, aa = o / uc;
          sA[u + LDC * aa] = left ? (A ? A[u0 + u + lda * aa] : 1.0) : A[i + nk * (u0 + u) + lda * aa];
        }
        for (int o = threadIdx.x; o < uc * rc; o += blockDim.x) {
          const int u = o % uc, cc = o / uc;
          sB[u + LDC * cc] = left ? B[u0 + u + inner * i + ldb * cc] : (B ? B[u0 + u + ldb * cc] : 1.0);
        }
        __syncthreads();
        if (sp < nsplit)
          for (int u = sp; u < uc; u += nsplit) acc = fma(sA[u + LDC * a], sB[u + LDC * c], acc);
      }
      red[threadIdx.x] = sp < nsplit ? acc : 0.0;
      __syncthreads();
      if ((int)threadIdx.x < Pg) {
        double t = 0.0;
        for (int q = 0; q < nsplit; ++q) t += red[threadIdx.x + Pg * q];
        Gi[a + rpa * nk * c] = t;
      }
      __syncthreads();
    }
    for (int o = threadIdx.x; o < rpa * rpc; o += blockDim.x) {
      const int a = o % rpa, c = o / rpa;
      if (a >= ra || c >= rc) Gi[a + rpa * nk * c] = 0.0;
    }
  }
}

// Large cores of a single problem in digit arithmetic: C(a, i, j) += sum_u A(u, a)
// B(u, i, j) over one K range of slice i (cores_kernel's products; FP64 FMAs bound
// those: 1.72 per cycle and SM on this GPU, against 1015 BF16 ones, which is 27 FP64
// products in the 37 digit products formed here).  A block takes 64 contraction
// indices at a time: a warp loads one column's 64 values (two per lane), scales
// them by the column's largest exponent in this chunk and writes their eight
// balanced base-256 digits (61 bits); every (16 a) x (8 j) tile sums its digit products
// of weight at most seven exactly in FP32 (8 x 64 x 2^14 < 2^24) and adds them to its
// FP64 sums.  The pairs left out are below 64 2^-57 of the two largest factors' product; where
// the factors' magnitudes say that this is not small against sum |A B| (digit::weak, one
// more product, of the leading digits without their signs), the 64 products are FP64 FMAs.
// So an entry is held to 2^-44 of sum |A B| at worst, and otherwise is closer than FP64 FMAs.
// Measured (middle core of 960^3, r = 25, l = 35): H = S M 1.64 ms and Q^T H 3.14 ms
// -> Q^T S 0.73 ms (0.60 with seven digits and no test of the terms) and (Q^T S) M 0.04.
struct CoreGemm {
  const double *A, *B;
  double* C;
  int64_t sau, lda, sai;    // A(u, a) of slice i at u sau + a lda + i sai
  int64_t ldb, sbi;         // B(u, i, j) at u + j ldb + i sbi
  int64_t ldc, sci;         // C(a, i, j) at a + i sci + j ldc
  int64_t inner, klen;      // contraction length, the part of one block
  int ra, rb;
};
constexpr int kGemmP = 8, kGemmK = 64;
// s + sum_u A(u sau) B(u) in FP64.
__device__ __noinline__ double core_dot(const double* A, int64_t sau, const double* B, int n, double s) {
#pragma unroll 8
  for (int u = 0; u < n; ++u) s = fma(A[u * sau], B[u], s);
  return s;
}
__global__ void __launch_bounds__(kThreads, 2) core_gemm_kernel(const CoreGemm g) {
  using namespace digit;
  constexpr int P = kGemmP, LEAD = 5, B = 8 * (P - 1) + LEAD, NW = P;   // weights kept: 0..7
  extern __shared__ __align__(16) double sm[];
  const int ma = (g.ra + 15) / 16, nb = (g.rb + 7) / 8, rows = 16 * ma + 8 * nb;
  uint16_t* D = reinterpret_cast<uint16_t*>(sm);             // [P][rows][kGemmK]: A's columns, then B's
  int* er = reinterpret_cast<int*>(D + P * rows * kGemmK);  // column exponents
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, gq = lane >> 2, tq = lane & 3;
  const int64_t i = blockIdx.x, k0 = (int64_t)blockIdx.y * g.klen, k1 = imin64(g.inner, k0 + g.klen);
  const double *Ai = g.A + g.sai * i, *Bi = g.B + g.sbi * i;
  const int tiles = ma * nb;
  double c[4][4];
#pragma unroll
  for (int q = 0; q < 4; ++q) c[q][0] = c[q][1] = c[q][2] = c[q][3] = 0.0;
  int bad = 0;
  for (int64_t u0 = k0; u0 < k1; u0 += kGemmK) {
    __syncthreads();
    for (int r0 = warp; r0 < rows; r0 += 4 * (kThreads / 32)) {
      double x[4][2];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int r = r0 + q * (kThreads / 32);
        const bool isa = r < 16 * ma;
        const int col = isa ? r : r - 16 * ma;
        const bool on = r < rows && col < (isa ? g.ra : g.rb);
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          const int64_t u = u0 + 2 * lane + e;
          x[q][e] = on && u < k1 ? (isa ? Ai[u * g.sau + col * g.lda] : Bi[u + col * g.ldb]) : 0.0;
        }
      }
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int r = r0 + q * (kThreads / 32);
        if (r >= rows) break;
        bad |= (undigital(x[q][0]) || undigital(x[q][1])) ? 1 : 0;
        const int m = __reduce_max_sync(0xffffffffu, max(exp_of(x[q][0]), exp_of(x[q][1])));
        if (lane == 0) er[r] = m;
        uint32_t d0[P], d1[P];
        digits<P>(fixed<B>(x[q][0], m), d0);
        digits<P>(fixed<B>(x[q][1], m), d1);
#pragma unroll
        for (int p = 0; p < P; ++p)
          *reinterpret_cast<uint32_t*>(D + (p * rows + r) * kGemmK + 8 * ((lane >> 2) ^ (r & 7)) + 2 * (lane & 3)) =
              d0[p] | (d1[p] << 16);
      }
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int t = warp + q * (kThreads / 32);
      if (t < tiles) {
        const int mt = t % ma, nt = t / ma;
        float acc[NW][4], mag[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int w = 0; w < NW; ++w) acc[w][0] = acc[w][1] = acc[w][2] = acc[w][3] = 0.0f;
        const uint32_t pa = s_u32(D + (16 * mt + (lane & 7) + 8 * ((lane >> 3) & 1)) * kGemmK);
        const uint32_t pb = s_u32(D + (16 * ma + 8 * nt + (lane & 7)) * kGemmK);
        const int stride = 2 * rows * kGemmK;   // bytes between digit arrays
#pragma unroll 1
        for (int kk = 0; kk < kGemmK / 8; kk += 4) {   // 16-byte chunks, swizzled by their row
          uint32_t fb[P][4];   // two k-steps of each digit of B
#pragma unroll
          for (int p = 0; p < P; ++p) ldsm4(pb + p * stride + 16 * ((kk + (lane >> 3)) ^ (lane & 7)), fb[p]);
#pragma unroll
          for (int ks = 0; ks < 2; ++ks)
#pragma unroll
            for (int p = 0; p < P; ++p) {
              uint32_t fa[4];
              ldsm4(pa + p * stride + 16 * ((kk + 2 * ks + (lane >> 4)) ^ (lane & 7)), fa);
              if (p == 0) mma_abs(mag, fa, fb[0] + 2 * ks);
#pragma unroll
              for (int p2 = 0; p2 < P; ++p2)
                if (p + p2 < NW) mma(acc[(p + p2) % NW], fa, fb[p2] + 2 * ks);
            }
        }
        uint32_t redo = 0;
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const int ea = er[16 * mt + gq + 8 * (e >> 1)], eb = er[16 * ma + 8 * nt + 2 * tq + (e & 1)];
          if (ea == kExpZero || eb == kExpZero) continue;   // a column of zeros
          if (weak(mag[e], 0x1p-5f, LEAD, c[q][e], ea + eb - 4)) {
            redo |= 1u << e;
            continue;
          }
          long long hi = 0, lo = 0;
#pragma unroll
          for (int w = 0; w < 4; ++w) {
            hi = hi * 256 + __float2int_rn(acc[w][e]);
            lo = lo * 256 + __float2int_rn(acc[w + 4][e]);
          }
          if (hi | lo) {   // (hi 2^32 + lo) 2^(ea + eb - 2 LEAD - 56)
            const int x = ea + eb - 2 * LEAD - 56;
            const double v = fma((double)hi, 4294967296.0, (double)lo);
            if (x > -900 && x < 900) c[q][e] = fma(v, __hiloint2double((x + 1023) << 20, 0), c[q][e]);
            else c[q][e] += ldexp(v, x);
          }
        }
#pragma unroll
        for (int e = 0; e < 4; ++e)
          if (redo >> e & 1) {
            const int a = 16 * mt + gq + 8 * (e >> 1), j = 8 * nt + 2 * tq + (e & 1);
            c[q][e] = core_dot(Ai + u0 * g.sau + a * g.lda, g.sau, Bi + u0 + j * g.ldb, (int)imin64(kGemmK, k1 - u0), c[q][e]);
          }
      }
    }
  }
  // a non-finite value in this block's range: its products as FP64 FMAs
  if (__syncthreads_or(bad)) {
    for (int o = threadIdx.x; o < g.ra * g.rb; o += kThreads) {
      const int a = o % g.ra, j = o / g.ra;
      double s = 0.0;
      for (int64_t u = k0; u < k1; ++u) s = fma(Ai[u * g.sau + a * g.lda], Bi[u + j * g.ldb], s);
      atomicAdd(g.C + a + g.sci * i + g.ldc * j, s);
    }
    return;
  }
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int t = warp + q * (kThreads / 32);
    if (t >= tiles) break;
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const int a = 16 * (t % ma) + gq + 8 * (e >> 1), j = 8 * (t / ma) + 2 * tq + (e & 1);
      if (a < g.ra && j < g.rb) atomicAdd(g.C + a + g.sci * i + g.ldc * j, c[q][e]);
    }
  }
}

// G(a, i, c) = sum_j T(a, i, j) M(j, c) (T: ra x n x l, M: l x rc with columns past
// the rank zero), one thread per entry.
__global__ void __launch_bounds__(kThreads) core_tm_kernel(const double* T, const double* M, double* G, int64_t rows,
                                                           int l, int rc) {
  __shared__ double Ms[TT_MAXL * TT_MAXL];
  for (int o = threadIdx.x; o < l * rc; o += blockDim.x) Ms[o] = M[o];
  __syncthreads();
  for (int64_t o = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; o < rows * rc; o += (int64_t)gridDim.x * blockDim.x) {
    const int64_t r = o % rows;
    const int c = (int)(o / rows);
    double s = 0.0;
    for (int j = 0; j < l; ++j) s = fma(T[r + rows * j], Ms[j + l * c], s);
    G[o] = s;
  }
}

// Two-pass middle core, eq. (3.5): G_{d*}(a, i, c) =
//   sum_{u, v} Q_{d*-1}(u, a) X(u + N_{d*-1} i + N_{d*} v) P_{d*}(v, c).
// One block per (i, chunk of v): y(v, a) = sum_u Q(u, a) X(...), then the
// block adds sum_v y(v, a) P(v, c) into the (zeroed) core with atomics.
__global__ void __launch_bounds__(kThreads) twopass_mid_kernel(char* wsb, const void* X, double* cores,
                                                               const int* ranks) {
  constexpr int CH = 64;
  __shared__ double Ys[CH * TT_MAXL];
  const DevItem& it = ditems(wsb)[0];
  const DevSketch* S = dsk(wsb);
  const double* ws = reinterpret_cast<const double*>(wsb);
  const int ds = it.ds;
  const int* rk = ranks + it.rank_off;
  const int ra = rk[ds - 1], rc = rk[ds];
  const int rpa = it.rpad[ds - 1];
  const int64_t Np = it.N[ds - 1], nk = it.n[ds - 1], Nm = it.N[ds];
  const int64_t Mm = it.N[it.d] / Nm;
  const double* Q = nullptr;
  int64_t ldq = 1;
  if (ds >= 2) {
    Q = ws + S[it.basis_of_k[ds - 1]].lev_z[0];
    ldq = S[it.basis_of_k[ds - 1]].rows;
  }
  const DevSketch& sp = S[it.basis_of_k[ds]];
  const double* Pm = ws + sp.lev_z[0];
  double* G = cores + it.core_off[ds];
  const int64_t nchunks = (Mm + CH - 1) / CH;
  for (int64_t job = blockIdx.x; job < nk * nchunks; job += gridDim.x) {
    const int64_t i = job % nk, v0 = (job / nk) * CH;
    const int nv = (int)imin64(CH, Mm - v0);
    __syncthreads();
    for (int o = threadIdx.x; o < CH * ra; o += blockDim.x) {
      const int v = o % CH, a = o / CH;
      double acc = 0.0;
      if (v < nv) {
        const int64_t base = Np * i + Nm * (v0 + v);
        for (int64_t u = 0; u < Np; ++u) {
          const double x = it.x_f64 ? ((const double*)X)[base + u] : (double)((const float*)X)[base + u];
          acc += (Q ? Q[u + ldq * a] : 1.0) * x;
        }
      }
      Ys[v + CH * a] = acc;
    }
    __syncthreads();
    for (int o = threadIdx.x; o < ra * rc; o += blockDim.x) {
      const int a = o % ra, c = o / ra;
      double acc = 0.0;
      for (int v = 0; v < nv; ++v) acc += Ys[v + CH * a] * Pm[v0 + v + sp.rows * c];
      atomicAdd(G + a + rpa * (i + nk * c), acc);
    }
  }
}

// One-sided two-pass last core (Algorithm 2): G_d(a, i, 0) = sum_u
// Q_{d-1}(u, a) X(u + N_{d-1} i).  Block (i, row chunk): the threads stride
// over the chunk's rows (coalesced in X and in each column of Q), eight
// columns a at a time with unconditional FMAs (columns past r_{d-1} read
// column r_{d-1} - 1 and are dropped), then a block sum and one atomic per a.
__global__ void __launch_bounds__(kThreads) twopass_last_kernel(char* wsb, const void* X, double* cores,
                                                                const int* ranks, int64_t chunk) {
  __shared__ double red[32];
  const DevItem& it = ditems(wsb)[0];
  const DevSketch& sq = dsk(wsb)[it.basis_of_k[it.d - 1]];
  const double* ws = reinterpret_cast<const double*>(wsb);
  const double* Q = ws + sq.lev_z[0];
  const int64_t ldq = sq.rows;
  const int ra = ranks[it.rank_off + it.d - 1];
  const int rpa = it.rpad[it.d - 1];
  const int64_t Np = it.N[it.d - 1];
  const int64_t i = blockIdx.x;
  const int64_t u0 = (int64_t)blockIdx.y * chunk, u1 = imin64(Np, u0 + chunk);
  double* G = cores + it.core_off[it.d];
  for (int a0 = 0; a0 < ra; a0 += 8) {
    double acc[8] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
    const double* qc[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) qc[j] = Q + ldq * min(a0 + j, ra - 1);
    for (int64_t u = u0 + threadIdx.x; u < u1; u += blockDim.x) {
      const int64_t e = u + Np * i;
      const double x = it.x_f64 ? reinterpret_cast<const double*>(X)[e] : (double)reinterpret_cast<const float*>(X)[e];
#pragma unroll
      for (int j = 0; j < 8; ++j) acc[j] = fma(qc[j][u], x, acc[j]);
    }
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const double t = block_sum(acc[j], red);
      if (threadIdx.x == 0 && a0 + j < ra) atomicAdd(G + (a0 + j) + (int64_t)rpa * i, t);
    }
  }
}

// Work from which a core goes to core_gemm_kernel (FMAs; 2^25 take cores_kernel
// 67 us at the FP64 pipe's rate, the three extra launches about 10).
constexpr int64_t kGemmMin = 1LL << 25;

// The one-pass middle core as (Q_{d*-1}^T S) M instead of Q_{d*-1}^T (S M): T = Q^T S is
// formed by core_gemm_kernel in H's place, and H itself is not needed (the backward
// forms it when it runs).  For large middle sketches that the region of H can
// hold T of.
bool mid_by_gemm(const Plan& P, int item) {
  const DevItem& it = plan_items_host(&P)[item];
  if (plan_num_items(&P) != 1 || it.passes != 1 || it.sided1 || it.ds < 2 || it.mcore != it.ds) return false;
  const int64_t ra = it.rpad[it.ds - 1], rc = it.rpad[it.ds], l = it.lmid;
  return ra * l * it.N[it.ds] >= kGemmMin && ra * l <= rc * (l + ra) && ra * l <= it.N[it.ds - 1] * rc;
}

cudaError_t run_core_gemm(CoreGemm g, int64_t n, int64_t nout, cudaStream_t st) {
  const int rows = (g.ra + 15) / 16 * 16 + (g.rb + 7) / 8 * 8;
  const size_t smem = 2ul * kGemmP * rows * kGemmK + sizeof(int) * rows;
  static bool attr = false;
  cudaError_t e;
  if (!attr) {
    e = cudaFuncSetAttribute(core_gemm_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)(2 * kGemmP * 2 * TT_MAXL * kGemmK + sizeof(int) * 2 * TT_MAXL));
    if (e != cudaSuccess) return e;
    attr = true;
  }
  e = cudaMemsetAsync(g.C, 0, sizeof(double) * nout, st);
  if (e != cudaSuccess) return e;
  // slices shorter than two blocks per SM are split along the contraction
  const int64_t split = std::max<int64_t>(1, std::min<int64_t>((2LL * device_sm_count() + n - 1) / n, g.inner / 256));
  g.klen = ((g.inner + split - 1) / split + kGemmK - 1) / kGemmK * kGemmK;
  count_launch();
  core_gemm_kernel<<<dim3((unsigned)n, (unsigned)((g.inner + g.klen - 1) / g.klen)), kThreads, smem, st>>>(g);
  return cudaGetLastError();
}

// The cores of a single problem that are large enough for core_gemm_kernel; their
// bits are set in *done.
cudaError_t launch_core_gemms(const Plan& P, void* ws, double* cores, uint32_t* done, cudaStream_t st) {
  const DevItem& it = plan_items_host(&P)[0];
  const DevSketch* S = plan_sketches_host(&P);
  double* W = (double*)ws;
  *done = 0;
  if (plan_num_items(&P) != 1 || it.sided1) return cudaSuccess;
  for (int k = 2; k < it.d; ++k) {
    const int64_t n = it.n[k - 1], ra = it.rpad[k - 1], rc = it.rpad[k];
    const bool left = k <= it.ds, mid = k == it.mcore;
    if (mid && !mid_by_gemm(P, 0)) continue;
    CoreGemm g;
    g.ra = (int)ra;
    g.rb = (int)(mid ? it.lmid : rc);
    g.inner = left ? it.N[k - 1] : it.N[it.d] / it.N[k];
    if (ra * g.rb * g.inner * n < kGemmMin || n >= (1LL << 31)) continue;
    const DevSketch& sa = S[it.basis_of_k[k - 1]];
    const DevSketch& sb = S[mid ? it.mid_sk : it.basis_of_k[k]];
    g.A = W + sa.lev_z[0];
    g.lda = sa.rows;
    g.sau = left ? 1 : n;
    g.sai = left ? 0 : 1;
    g.B = W + (mid ? sb.off : sb.lev_z[0]);
    g.ldb = sb.rows;
    g.sbi = left ? g.inner : 0;
    g.C = mid ? W + it.off_H : cores + it.core_off[k];
    g.sci = ra;
    g.ldc = ra * n;
    cudaError_t e = run_core_gemm(g, n, ra * n * g.rb, st);
    if (e != cudaSuccess) return e;
    if (mid) {
      const int64_t rows = ra * n;
      const int grid = (int)std::min<int64_t>((rows * rc + kThreads - 1) / kThreads, 16LL * device_sm_count());
      count_launch();
      core_tm_kernel<<<grid, kThreads, 0, st>>>(g.C, W + it.off_QB, cores + it.core_off[k], rows, it.lmid, (int)rc);
      e = cudaGetLastError();
      if (e != cudaSuccess) return e;
    }
    *done |= 1u << k;
  }
  return cudaSuccess;
}

cudaError_t launch_mid_h(const Plan& P, int item, void* ws, const int* ranks, cudaStream_t st) {
  const DevItem& it = plan_items_host(&P)[item];
  const int64_t Nm = plan_sketches_host(&P)[it.mid_sk].rows;
  const int grid = (int)std::min<int64_t>((Nm * it.rpad[it.mbk] + kThreads - 1) / kThreads, 8LL * device_sm_count());
  count_launch();
  mid_h_kernel<<<grid, kThreads, 0, st>>>((char*)ws, item, ranks);
  return cudaGetLastError();
}

}  // namespace

// H for the backward, when the forward's middle core did without it.
cudaError_t launch_backward_h(const Plan& P, int item, void* ws, const int* ranks, cudaStream_t st) {
  return mid_by_gemm(P, item) ? launch_mid_h(P, item, ws, ranks, st) : cudaSuccess;
}

cudaError_t launch_mid_b_mixed(const Plan& P, int item, void* ws, const int* ranks, cudaStream_t st);

// Dynamic shared memory of mid_ls_kernel.
size_t ls_smem(int l, int r) { return sizeof(double) * ((size_t)qr_ld(l) * r + (size_t)(l + 1) * r); }

// Middle cores of every item of a batched plan; B was zeroed with the sketches.
cudaError_t launch_finalize_mid_batched(const Plan& P, void* ws, const int* ranks, cudaStream_t st) {
  char* wsb = (char*)ws;
  const int nitems = plan_num_items(&P);
  const DevSketch* sks = plan_sketches_host(&P);
  int64_t Mmax = 1, Nmax = 1;
  int lmax = 1, rmax = 1;
  for (int i = 0; i < nitems; ++i) {
    const DevItem& it = plan_items_host(&P)[i];
    Mmax = std::max(Mmax, sks[it.basis_of_k[it.mbk]].rows);
    Nmax = std::max(Nmax, sks[it.mid_sk].rows);
    lmax = std::max(lmax, it.lmid);
    rmax = std::max(rmax, it.rpad[it.mbk]);
  }
  cudaError_t e;
  if (plan_items_host(&P)[0].prec == TT_PREC_FP64) {
    const unsigned gx = (unsigned)std::min<int64_t>((Mmax + 31) / 32, 64);
    count_launch();
    mid_b_kernel_f64<<<dim3(gx, (unsigned)nitems), kThreads, 0, st>>>(wsb, -1, ranks);
    e = cudaGetLastError();
  } else {
    e = launch_mid_b_mixed_batched(P, ws, ranks, st);
  }
  if (e != cudaSuccess) return e;
  count_launch();
  mid_ls_kernel<<<dim3(1, (unsigned)nitems), kThreads, ls_smem(lmax, rmax), st>>>(wsb, -1, ranks);
  e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  const unsigned gx = (unsigned)std::min<int64_t>((Nmax * TT_MAXL + kThreads - 1) / kThreads, 64);
  count_launch();
  mid_h_kernel<<<dim3(gx, (unsigned)nitems), kThreads, 0, st>>>(wsb, -1, ranks);
  return cudaGetLastError();
}

cudaError_t launch_finalize(const Plan& P, void* ws, double* cores, int* ranks, cudaStream_t st) {
  char* wsb = (char*)ws;
  const int max_lev = plan_max_lev(&P);
  const DevSketch* sks = plan_sketches_host(&P);
  const int nitems = plan_num_items(&P);
  cudaError_t e;
  if (nitems == 1) {  // the slab kernel's staged S_2 partials not yet folded
    e = fold_s2_staging(P, 0, ws, st);
    if (e != cudaSuccess) return e;
  }
  static bool attr = false;
  if (!attr) {
    e = cudaFuncSetAttribute(tsqr_level_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kTsqrSmemMax);
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(tsqr_expand_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kTsqrSmemMax);
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(mid_ls_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)ls_smem(TT_MAXL, TT_MAXL));
    if (e != cudaSuccess) return e;
    attr = true;
  }
  // FP16 items: sketches back to the scale of X, and the range check
  {
    bool any16 = false;
    for (int i = 0; i < nitems; ++i) any16 = any16 || plan_items_host(&P)[i].prec == TT_PREC_FP16;
    if (any16) {
      count_launch();
      sketch_unscale_kernel<<<dim3((unsigned)(4 * device_sm_count()), (unsigned)nitems), kThreads, 0, st>>>(wsb, 0);
      e = cudaGetLastError();
      if (e != cudaSuccess) return e;
    }
  }
  int maxw = 1, maxr = 1;
  for (int i = 0, n = 0; i < nitems; ++i) {
    const DevItem& it = plan_items_host(&P)[i];
    for (int s = 0; s < it.nsk; ++s) {
      const DevSketch& d = sks[it.sk0 + s];
      if (!d.basis) continue;
      maxw = std::max(maxw, d.width);
      maxr = std::max(maxr, d.rpad);
      ++n;
    }
  }
  // shared memory of each level's launch (the trees are aligned at their roots)
  size_t smem_up[kMaxLev] = {}, smem_down[kMaxLev] = {};
  for (int i = 0; i < nitems; ++i) {
    const DevItem& it = plan_items_host(&P)[i];
    for (int s = 0; s < it.nsk; ++s) {
      const DevSketch& d = sks[it.sk0 + s];
      if (!d.basis) continue;
      for (int L = 0; L < d.nlev; ++L) {
        const int g = L + max_lev - d.nlev;
        smem_up[g] = std::max(smem_up[g], (size_t)(sizeof(double) * tsqr_block_doubles(d.lev_bl[L], d.width)));
        smem_down[g] = std::max(smem_down[g], sizeof(double) * ((size_t)tsqr_ld(d.lev_bl[L]) * d.width + TT_MAXL));
      }
    }
  }
  // the roots' expansion as a launch of its own, its columns over several CTAs, when
  // it is long enough to pay for the launch
  const int root_sep = nitems == 1 && maxr > 8 ? 1 : 0;
  for (int L = 0; L < max_lev; ++L) {
    const int nt = plan_ntasks(&P, L);
    if (nt == 0) continue;
    count_launch();
    tsqr_level_kernel<<<nt, kThreads, smem_up[L], st>>>(wsb, L, ranks, root_sep);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  for (int L = root_sep ? max_lev - 1 : max_lev - 2; L >= 0; --L) {
    const int nt = plan_ntasks(&P, L);
    if (nt == 0) continue;
    // columns per CTA: eight (one per warp) when the blocks alone leave SMs idle
    const int cw = nt * ((maxr + 7) / 8) <= 2 * device_sm_count() ? 8 : nt <= device_sm_count() ? 16 : TT_MAXL;
    count_launch();
    tsqr_expand_kernel<<<dim3((unsigned)nt, (unsigned)((maxr + cw - 1) / cw)), kThreads, smem_down[L], st>>>(wsb, L, ranks,
                                                                                                    root_sep, cw);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  // one-pass middle cores (one launch per step over all items when batched)
  if (nitems > 1) {
    e = launch_finalize_mid_batched(P, ws, ranks, st);
    if (e != cudaSuccess) return e;
  }
  for (int i = 0; i < nitems && nitems == 1; ++i) {
    const DevItem& it = plan_items_host(&P)[i];
    if (it.passes != 1) continue;
    const int rp = it.rpad[it.mbk];
    e = cudaMemsetAsync((double*)ws + it.off_B, 0, sizeof(double) * rp * it.lmid, st);
    if (e != cudaSuccess) return e;
    if (it.prec == TT_PREC_FP64) {
      const int64_t M = sks[it.basis_of_k[it.mbk]].rows;
      const int grid = (int)std::min<int64_t>((M + 31) / 32, 2LL * device_sm_count());
      count_launch();
      mid_b_kernel_f64<<<grid, kThreads, 0, st>>>(wsb, i, ranks);
      e = cudaGetLastError();
    } else {
      e = launch_mid_b_mixed(P, i, ws, ranks, st);
    }
    if (e != cudaSuccess) return e;
    count_launch();
    mid_ls_kernel<<<1, kThreads, ls_smem(it.lmid, it.rpad[it.mbk]), st>>>(wsb, i, ranks);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    if (!mid_by_gemm(P, i)) {
      e = launch_mid_h(P, i, ws, ranks, st);
      if (e != cudaSuccess) return e;
    }
  }
  uint32_t skip = 0;
  if (nitems == 1) {
    e = launch_core_gemms(P, ws, cores, &skip, st);
    if (e != cudaSuccess) return e;
  }
  int dmax = 1;
  int64_t nmax = 1;
  for (int i = 0; i < nitems; ++i) {
    const DevItem& it = plan_items_host(&P)[i];
    dmax = std::max(dmax, it.d);
    for (int k = 0; k < it.d; ++k) nmax = std::max(nmax, it.n[k]);
  }
  const int64_t gy = std::min<int64_t>(nmax, std::max<int64_t>(1, kCoreBlocks / ((int64_t)nitems * dmax)));
  dim3 grid((unsigned)(nitems * dmax), (unsigned)gy);
  count_launch();
  cores_kernel<<<grid, kThreads, 0, st>>>(wsb, cores, ranks, 0, nitems, 0, dmax, skip);
  return cudaGetLastError();
}

// Cores of one item only (k = only_k), used by the two-pass middle core.
cudaError_t launch_cores_one(const Plan& P, int item, int only_k, void* ws, double* cores,
                             const int* ranks, cudaStream_t st) {
  const DevItem& it = plan_items_host(&P)[item];
  dim3 grid((unsigned)it.d, (unsigned)std::min<int64_t>(it.n[only_k - 1], 512));
  count_launch();
  cores_kernel<<<grid, kThreads, 0, st>>>((char*)ws, cores, ranks, item, 1, only_k, it.d, 0u);
  return cudaGetLastError();
}

}  // namespace tts

namespace tts {
cudaError_t launch_twopass_mid(const Plan& P, const void* X, void* ws, double* cores, const int* ranks,
                               cudaStream_t st) {
  const DevItem& it = plan_items_host(&P)[0];
  if (it.sided1) {  // the last core G_d = Q_{d-1}^T X_{d-1}
    const int d = it.d;
    cudaError_t e = cudaMemsetAsync(cores + it.core_off[d], 0, sizeof(double) * it.rpad[d - 1] * it.n[d - 1], st);
    if (e != cudaSuccess) return e;
    const int64_t Np = it.N[d - 1], chunk = 65536;
    const dim3 grid((unsigned)it.n[d - 1], (unsigned)((Np + chunk - 1) / chunk));
    count_launch();
    twopass_last_kernel<<<grid, kThreads, 0, st>>>((char*)ws, X, cores, ranks, chunk);
    return cudaGetLastError();
  }
  const int ds = it.ds;
  cudaError_t e = cudaMemsetAsync(cores + it.core_off[ds], 0,
                                  sizeof(double) * it.rpad[ds - 1] * it.n[ds - 1] * it.rpad[ds], st);
  if (e != cudaSuccess) return e;
  const int64_t Mm = it.N[it.d] / it.N[ds];
  const int64_t jobs = it.n[ds - 1] * ((Mm + 63) / 64);
  const int grid = (int)std::min<int64_t>(jobs, 8LL * device_sm_count());
  count_launch();
  twopass_mid_kernel<<<grid, kThreads, 0, st>>>((char*)ws, X, cores, ranks);
  return cudaGetLastError();
}
}  // namespace tts
