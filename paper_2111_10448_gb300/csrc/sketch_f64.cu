// FP64 fused multi-sketch (the correctness path of the sketch step, Sec. 3.2
// and Algorithm 5: one read of each tile of X feeds every sketch).
//
// X is seen as planes X(:, w, :) (n_1 x n_d, see internal.cuh).  A work item is
// one tile (a-block x b-block) of one plane; it is staged in shared memory
// once, then every sketch adds its contribution:
//   column sketch: S_k[a + n_1 wlo, j] += sum_b X(a, w, b) Omega_k[whi + hs b, j]
//   row sketch:    R_k[whi + hs b, j]  += sum_a X(a, w, b) Psi_k[a + n_1 wlo, j]
// with the test-matrix tile regenerated from Philox into shared memory.  The
// per-tile partial sums are added to the FP64 sketches with atomics.
//
// What bounds it: the FP64 units (1.7 FMAs per cycle and SM measured), by the products
// and as much again by drawing the test-matrix rows, whose logarithms, roots and sines
// are FP64 too: a quad of normals costs as much as some 90 FMAs.  So rows that
// many tiles share are drawn once per accumulate into the backward's scratch (st_tab)
// and read from there, and planes wide enough take 64 x 64 tiles, which halves what is
// left on the row side.  Accumulate at 64^4, l = 50: 11.1 ms
// with every row drawn by every 64 x 32 tile, now 7.4, of which the products' FMAs are 6.7;
// 40^4, l = 16: 1.00 -> 0.49 ms; 300 x 200 x 100, l = 30: 2.18 -> 1.24.
#include <algorithm>

#include "internal.cuh"
#include "philox.cuh"
#include "testmat.cuh"

namespace tts {
const DevSketch* plan_sketches_host(const Plan* p);
namespace {

constexpr int64_t kTableOffB = 256;
constexpr int kTA = 64;   // rows (i_1) per tile of the single-tensor launch
constexpr int kTB = 32;   // columns (i_d) per tile
constexpr int kThreads = 256;
constexpr int64_t kGroupDoubles = 4096;    // rows of a group of sketches: 32 KB beside a tile of at most 33
constexpr int64_t kTableQuads = 1 << 17;   // quads of normals that pay for staging them (some 4 us of a launch)

struct SkArg {
  int64_t rows, off, wdiv, hstride;
  int type, width, sid;
  int kr;  // global sketch index when the test matrix is Khatri-Rao, -1: dense
  const double* tab;  // its staged rows (width doubles each), nullptr: drawn per tile
};

struct F64Args {
  const void* X;
  double* ws;
  int64_t n1, cnt, first, W, Nd1;
  uint64_t seed;
  int x_f64, nsk;
  SkArg sk[kMaxSk];
};

__device__ __forceinline__ double load_x(const void* X, int x_f64, int64_t i) {
  return x_f64 ? __ldg((const double*)X + i) : (double)__ldg((const float*)X + i);
}

template <int TA, int TB>
__host__ __device__ constexpr int64_t f64_tiles(int64_t W, int64_t n1, int64_t cnt) {
  return W * ((n1 + TA - 1) / TA) * ((cnt + TB - 1) / TB);
}

// One tile (TA rows of i_1 x TB columns of i_d of plane w) into every sketch.  The
// sketches go in groups whose rows fit gcap doubles together: a small tile has work
// for a few warps in each sketch only, and each is a chain of FP64 latencies, so
// the threads take the quads, then the products, of a whole group at once (40^4, l = 16:
// 0.72 -> 0.49 ms; 7 x 9 x 8 x 5 x 6, l = 8: 88 -> 54 us).
template <int TA, int TB>
__device__ void f64_tile(const F64Args& a, int64_t item, double* smem, int gcap) {
  constexpr int LDX = TA + 1;
  double* Xs = smem;                         // LDX x TB
  double* Gs = smem + LDX * TB;              // gcap: per sketch of a group, nr rows x (width + 1)
  const int tid = threadIdx.x;
  const int64_t nA = (a.n1 + TA - 1) / TA;
  const int64_t nB = (a.cnt + TB - 1) / TB;
  const int64_t w = item / (nA * nB);
  const int64_t rem = item - w * nA * nB;
  const int64_t bb = rem / nA, ab = rem - bb * nA;
  const int64_t a0 = ab * TA, b0 = bb * TB;
  const int ta = (int)imin64(TA, a.n1 - a0);
  const int tb = (int)imin64(TB, a.cnt - b0);
  __syncthreads();
  for (int o = tid; o < ta * tb; o += kThreads) {
    const int ib = o / ta, ia = o - ib * ta;
    Xs[ia + LDX * ib] = load_x(a.X, a.x_f64, (a0 + ia) + a.n1 * w + a.Nd1 * (b0 + ib));
  }
  for (int s0 = 0; s0 < a.nsk;) {
    int s1 = s0, used = 0;
    do {
      used += (a.sk[s1].type == SK_COL ? tb : ta) * (a.sk[s1].width + 1);
      ++s1;
    } while (s1 < a.nsk && used + (a.sk[s1].type == SK_COL ? tb : ta) * (a.sk[s1].width + 1) <= gcap);
    if (s0) __syncthreads();   // the products of the group before
    // test-matrix rows: sketch s's jobs follow those of s - 1 over the threads
    int base = 0;
    double* G = Gs;
    for (int s = s0; s < s1; ++s) {
      const SkArg& sk = a.sk[s];
      const int l = sk.width, LDG = l + 1, nr = sk.type == SK_COL ? tb : ta, nq = (l + 3) / 4;
      const int64_t wlo = w % sk.wdiv, whi = w / sk.wdiv;
      const int first = (tid - base) & (kThreads - 1);
      if (sk.tab) {
        // rows (whi, b0 ...) of a column sketch, (wlo, a0 ...) of a row sketch: consecutive
        const double* src = sk.tab + (sk.type == SK_COL ? whi * a.cnt + b0 : wlo * a.n1 + a0) * l;
        for (int o = first; o < nr * l; o += kThreads) {
          const int r = o / l;
          G[r * LDG + (o - r * l)] = src[o];
        }
        base += nr * l;
      } else {
        for (int o = first; o < nr * nq; o += kThreads) {
          const int q = o / nr, r = o - q * nr;
          const uint64_t grow = sk.type == SK_COL ? (uint64_t)(whi + sk.hstride * (a.first + b0 + r))
                                                  : (uint64_t)((a0 + r) + a.n1 * wlo);
          double z[4];
          tm_quad_f64(a.ws, kr_of(a.ws, sk.kr), a.seed, (uint32_t)sk.sid, grow, (uint32_t)q, z);
#pragma unroll
          for (int t = 0; t < 4; ++t)
            if (4 * q + t < l) G[r * LDG + 4 * q + t] = z[t];
        }
        base += nr * nq;
      }
      G += nr * LDG;
    }
    __syncthreads();
    base = 0;
    G = Gs;
    for (int s = s0; s < s1; ++s) {
      const SkArg& sk = a.sk[s];
      const int l = sk.width, LDG = l + 1;
      const int64_t wlo = w % sk.wdiv, whi = w / sk.wdiv;
      const int first = (tid - base) & (kThreads - 1);
      double* out = a.ws + sk.off;
      if (sk.type == SK_COL) {
        for (int o = first; o < ta * l; o += kThreads) {
          const int j = o / ta, ia = o - j * ta;
          double acc = 0.0;
          for (int ib = 0; ib < tb; ++ib) acc = fma(Xs[ia + LDX * ib], G[ib * LDG + j], acc);
          atomicAdd(out + (a0 + ia + a.n1 * wlo) + sk.rows * j, acc);
        }
        base += ta * l;
        G += tb * LDG;
      } else {
        for (int o = first; o < tb * l; o += kThreads) {
          const int j = o / tb, ib = o - j * tb;
          double acc = 0.0;
          for (int ia = 0; ia < ta; ++ia) acc = fma(Xs[ia + LDX * ib], G[ia * LDG + j], acc);
          atomicAdd(out + (whi + sk.hstride * (a.first + b0 + ib)) + sk.rows * j, acc);
        }
        base += tb * l;
        G += ta * LDG;
      }
    }
    s0 = s1;
  }
}

// gcap: doubles for the rows of one group of sketches, at least one sketch's.
template <int TA, int TB>
__host__ __device__ constexpr int f64_gcap(int lmax) {
  return (TA > TB ? TA : TB) * (lmax + 1);
}
template <int TA, int TB>
__host__ __device__ constexpr size_t f64_smem(int gcap) {
  return sizeof(double) * ((size_t)(TA + 1) * TB + (size_t)gcap);
}

template <int TB>
__global__ void __launch_bounds__(kThreads) sketch_f64_kernel(const __grid_constant__ F64Args a, int gcap) {
  extern __shared__ double smem[];
  const int64_t total = f64_tiles<kTA, TB>(a.W, a.n1, a.cnt);
  for (int64_t item = blockIdx.x; item < total; item += gridDim.x) f64_tile<kTA, TB>(a, item, smem, gcap);
}

// Rows (key, r), r < nr, of sketch s into its table: the test-matrix row key + hstride
// (first + r) of a column sketch, r + n_1 key of a row sketch.
__global__ void __launch_bounds__(256) f64_table_kernel(const F64Args a, int s, int64_t nkeys, int nr, double* tab) {
  const SkArg sk = a.sk[s];
  const int nq = (sk.width + 3) / 4;
  const int64_t total = nkeys * nr * nq;
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < total; e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t row = e / nq, key = row / nr;
    const int q = (int)(e - row * nq), r = (int)(row - key * nr);
    const uint64_t grow = sk.type == SK_COL ? (uint64_t)(key + sk.hstride * (a.first + r)) : (uint64_t)(r + a.n1 * key);
    double z[4];
    tm_quad_f64(a.ws, kr_of(a.ws, sk.kr), a.seed, (uint32_t)sk.sid, grow, (uint32_t)q, z);
#pragma unroll
    for (int t = 0; t < 4; ++t)
      if (4 * q + t < sk.width) tab[row * sk.width + 4 * q + t] = z[t];
  }
}

// Batched form: one persistent launch over the tiles of every tensor of the
// plan.  The tensors are visited in the plan's cost order (largest first) and
// their tiles numbered consecutively (prefix[] = first tile of each); a CTA
// takes `chunk` consecutive tiles at a time from a global counter.
template <int TA, int TB>
__global__ void __launch_bounds__(kThreads) sketch_f64_batched_kernel(const BatchLaunch b, int gcap) {
  extern __shared__ double smem[];
  __shared__ F64Args sa;
  __shared__ int64_t s_base;
  __shared__ int s_pos;
  const DevTables& T = *reinterpret_cast<const DevTables*>(b.wsb + kTableOffB);
  const DevItem* items = reinterpret_cast<const DevItem*>(b.wsb + T.off_items);
  const DevSketch* sks = reinterpret_cast<const DevSketch*>(b.wsb + T.off_sketches);
  const int* order = reinterpret_cast<const int*>(b.wsb + T.off_border);
  const int64_t* prefix = reinterpret_cast<const int64_t*>(b.wsb + T.off_bprefix);
  unsigned long long* counter = reinterpret_cast<unsigned long long*>(b.wsb + T.off_bcounter);
  const int64_t total = prefix[T.nitems];
  int cur = -1;
  for (;;) {
    if (threadIdx.x == 0) {
      s_base = (int64_t)atomicAdd(counter, (unsigned long long)b.chunk);
      // position of the tensor holding tile s_base (last prefix <= s_base)
      int lo = 0, hi = T.nitems - 1;
      if (s_base < total) {
        while (lo < hi) {
          const int mid = (lo + hi + 1) >> 1;
          if (prefix[mid] <= s_base) lo = mid;
          else hi = mid - 1;
        }
      }
      s_pos = lo;
    }
    __syncthreads();
    const int64_t base = s_base;
    int pos = s_pos;
    if (base >= total) break;
    const int64_t end = imin64(base + b.chunk, total);
    for (int64_t t = base; t < end; ++t) {
      while (prefix[pos + 1] <= t) ++pos;
      const int it_idx = order[pos];
      if (it_idx != cur) {
        __syncthreads();
        if (threadIdx.x == 0) {
          const DevItem& it = items[it_idx];
          sa.X = b.X[it_idx];
          sa.ws = reinterpret_cast<double*>(b.wsb);
          sa.n1 = it.n[0];
          sa.cnt = it.n[it.d - 1];
          sa.first = 0;
          sa.W = it.W;
          sa.Nd1 = it.N[it.d - 1];
          sa.seed = it.seed;
          sa.x_f64 = it.x_f64;
          sa.nsk = it.nsk;
          for (int s = 0; s < it.nsk; ++s) {
            const DevSketch& d = sks[it.sk0 + s];
            sa.sk[s] = SkArg{d.rows, d.off, d.wdiv, d.hstride, d.type, d.width, d.stream_id, -1, nullptr};
          }
        }
        __syncthreads();
        cur = it_idx;
      }
      f64_tile<TA, TB>(sa, t - prefix[pos], smem, gcap);
    }
    __syncthreads();
  }
}

}  // namespace

cudaError_t launch_sketch_f64(const Plan& P, int item, const void* X, int64_t first, int64_t count,
                              void* ws, cudaStream_t st) {
  const DevItem& it = plan_items_host(&P)[item];
  F64Args a;
  a.X = X;
  a.ws = (double*)ws;
  a.n1 = it.n[0];
  a.cnt = count;
  a.first = first;
  a.W = it.W;
  a.Nd1 = it.N[it.d - 1];
  a.seed = it.seed;
  a.x_f64 = it.x_f64;
  a.nsk = it.nsk;
  const DevSketch* sks = plan_sketches_host(&P);
  int lmax = 1;
  for (int s = 0; s < it.nsk; ++s) {
    const DevSketch& d = sks[it.sk0 + s];
    a.sk[s] = SkArg{d.rows, d.off, d.wdiv, d.hstride, d.type, d.width, d.stream_id, d.kr_nm ? it.sk0 + s : -1, nullptr};
    lmax = d.width > lmax ? d.width : lmax;
  }
  // 64 columns a tile where the planes have them and the tiles still fill the SMs
  const bool wide = count > kTB && f64_tiles<kTA, 64>(a.W, a.n1, count) >= 4LL * device_sm_count();
  const int64_t nA = (a.n1 + kTA - 1) / kTA, nB = wide ? (count + 63) / 64 : (count + kTB - 1) / kTB;
  for (int s = 0; s < it.nsk; ++s) {
    const DevSketch& d = sks[it.sk0 + s];
    if (d.st_tab < 0) continue;
    // rows staged once and the rows drawn by the tiles otherwise; a launch costs as much
    // as kTableQuads drawn quads
    const bool col = d.type == SK_COL;
    const int64_t nkeys = col ? it.W / d.wdiv : d.wdiv, nr = col ? count : a.n1;
    const int64_t uses = col ? d.wdiv * nA : (it.W / d.wdiv) * nB, nq = (d.width + 3) / 4;
    if (nr >= (1LL << 31) || (uses - 1) * nkeys * nr * nq < kTableQuads) continue;
    double* tab = (double*)((char*)ws + d.st_tab);
    const int64_t blocks = std::min<int64_t>((nkeys * nr * nq + 255) / 256, 8LL * device_sm_count());
    count_launch();
    f64_table_kernel<<<(unsigned)blocks, 256, 0, st>>>(a, s, nkeys, (int)nr, tab);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    a.sk[s].tab = tab;
  }
  // the rows of all sketches in one group where they are few
  int64_t all = 0;
  for (int s = 0; s < it.nsk; ++s)
    all += std::min<int64_t>(a.sk[s].type == SK_COL ? count : a.n1, a.sk[s].type == SK_COL && !wide ? kTB : 64) *
           (a.sk[s].width + 1);
  const int gcap = (int)std::max<int64_t>(wide ? f64_gcap<kTA, 64>(lmax) : f64_gcap<kTA, kTB>(lmax),
                                          std::min<int64_t>(all, kGroupDoubles));
  const size_t smem = wide ? f64_smem<kTA, 64>(gcap) : f64_smem<kTA, kTB>(gcap);
  const auto kern = wide ? sketch_f64_kernel<64> : sketch_f64_kernel<kTB>;
  static bool attr_set[2] = {false, false};
  if (!attr_set[wide]) {
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, 96 * 1024);
    if (e != cudaSuccess) return e;
    attr_set[wide] = true;
  }
  const int64_t grid = std::min<int64_t>(a.W * nA * nB, (1LL << 31) - 1);   // a CTA per tile: no uneven last share
  count_launch();
  kern<<<(unsigned)grid, kThreads, smem, st>>>(a, gcap);
  return cudaGetLastError();
}

int64_t batched_tiles_f64(int64_t W, int64_t n1, int64_t cnt, int ta) {
  return ta == 32 ? f64_tiles<32, kTB>(W, n1, cnt) : f64_tiles<64, kTB>(W, n1, cnt);
}

cudaError_t launch_sketch_f64_batched(const BatchLaunch& b, const BatchCfg& cfg, int lmax, cudaStream_t st) {
  const int gcap = cfg.ta == 32 ? f64_gcap<32, kTB>(lmax) : f64_gcap<64, kTB>(lmax);
  const size_t smem = cfg.ta == 32 ? f64_smem<32, kTB>(gcap) : f64_smem<64, kTB>(gcap);
  auto kern = cfg.ta == 32 ? sketch_f64_batched_kernel<32, kTB> : sketch_f64_batched_kernel<64, kTB>;
  static bool attr_set[2] = {false, false};
  if (!attr_set[cfg.ta == 32]) {
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, 96 * 1024);
    if (e != cudaSuccess) return e;
    attr_set[cfg.ta == 32] = true;
  }
  count_launch();
  kern<<<cfg.ctas_per_sm * device_sm_count(), kThreads, smem, st>>>(b, gcap);
  return cudaGetLastError();
}

}  // namespace tts
