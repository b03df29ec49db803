// Strip kernel: launch arguments and the device code of one operand format;
// sketch_strip_<format>.cu instantiate it, sketch_strip.cu plans the launch.
//
// The fused multi-sketch (BF16, FP16 or TF32 tensor cores, X split into hi +
// lo) for every shape that neither the tcgen05 kernels nor the small-plane
// kernel take.  See sketch_strip.cu for the split of the work.
#pragma once
#include <cstdint>

#include "internal.cuh"
#include "philox.cuh"
#include "tc_common.cuh"
#include "testmat.cuh"

namespace tts {
namespace strip {

constexpr int kThreads = 256, kWarps = 8;
constexpr int kMaxCol = 3, kMaxRow = 3;   // sketches a side
constexpr int kMaxTA = 128;               // rows of i_1 per strip: one 16-row m-tile per warp
constexpr int kMaxTasks = 8 * kMaxRow;    // row products (m-tile, sketch) of one tile
constexpr int kAddsMax = 32;              // FP32 additions into one accumulator between FP64 flushes
constexpr int kRowAddsMax = 16;           // the same for the row sketches' shared sums (4 chunks each)
constexpr int kFmtBF16 = 0, kFmtTF32 = 1, kFmtFP16 = 2;

__host__ __device__ constexpr int esz(int fmt) { return fmt == kFmtTF32 ? 4 : 2; }
// Bytes of a staged test-matrix row of NT column octets.  16-bit rows are an
// odd number of 16-byte chunks, so that the eight row addresses of an ldmatrix
// fall on distinct banks; TF32 rows are 8 or 24 words past a multiple of 32, so
// that the four k rows of a fragment load do.
__host__ __device__ constexpr int ldg_bytes(int fmt, int nt) {
  return fmt == kFmtTF32 ? (nt * 8 + ((nt & 1) ? 0 : 8)) * 4 : (nt | 1) * 16;
}

struct StSk {
  int64_t rows, off, hstride;
  int64_t tab;          // byte offset (from the workspace base) of the staged rows, -1: generated
  uint32_t wdiv;        // N_k / n_1
  int width, lpad, sid;
  int kr;               // global sketch index when the test matrix is Khatri-Rao, -1: dense
  int mbm;              // mode-by-mode Khatri-Rao sketch (scaled per plane)
  int soff;             // byte offset of its staged block in shared memory
};

struct StripArgs {
  const float* X;
  char* wsb;
  int64_t n1, cnt, first, Nd1;
  uint64_t seed;
  uint32_t WL, WR, q2, q3;    // kL = i_2 + q2 i_3 (q2 q3 = WL)
  int ncol, nrow, vec;
  float xscale;
  int nA, TA, nB, TB;         // strips of i_1 and tiles of i_d
  uint32_t ngt;               // column tiles (kR, i_d block): WR nB
  int NG, nGS;                // column tiles per unit, sets of them
  uint32_t CL;                // kL values per unit
  uint32_t inv_qpr, inv_cpr;  // reciprocals (20 bits) of TA / 4 and of the copied chunks a row
  int cpr;                    // 16-byte chunks copied per row: TA / 4, one more for unaligned rows
  int off_xl, off_raw, off_acc, off_scale;   // shared-memory byte offsets
  int64_t total;              // entries of the slab (bounds of the 16-byte copies)
  StSk col[kMaxCol], row[kMaxRow];
  uint8_t task[kWarps][kMaxTasks];  // row products of each warp: m-tile + 8 sketch, 255 ends the list
};

__device__ __forceinline__ uint32_t s_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void ldsm4(uint32_t a, uint32_t* r) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(a));
}
__device__ __forceinline__ void ldsm4t(uint32_t a, uint32_t* r) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(a));
}
__device__ __forceinline__ void ldsm2t(uint32_t a, uint32_t* r) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x2.trans.shared.b16 {%0,%1}, [%2];" : "=r"(r[0]), "=r"(r[1]) : "r"(a));
}
__device__ __forceinline__ float lds_f(uint32_t a) {
  float v;
  asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(a));
  return v;
}
// c = a b (+ c unless FIRST).
#define TT_STRIP_MMA(SHAPE, TYPES)                                                                             \
  if constexpr (FIRST)                                                                                         \
    asm volatile("mma.sync.aligned." SHAPE ".row.col.f32." TYPES ".f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, " \
                 "{%10,%10,%10,%10};" : "=f"(c[0]), "=f"(c[1]), "=f"(c[2]), "=f"(c[3])                          \
                 : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]), "f"(0.0f));                \
  else                                                                                                         \
    asm volatile("mma.sync.aligned." SHAPE ".row.col.f32." TYPES ".f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, " \
                 "{%0,%1,%2,%3};" : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])                              \
                 : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]))
template <int FMT, bool FIRST>
__device__ __forceinline__ void mma(float* c, const uint32_t* a, const uint32_t* b) {
  if constexpr (FMT == kFmtBF16) {
    TT_STRIP_MMA("m16n8k16", "bf16.bf16");
  } else if constexpr (FMT == kFmtFP16) {
    TT_STRIP_MMA("m16n8k16", "f16.f16");
  } else {
    TT_STRIP_MMA("m16n8k8", "tf32.tf32");
  }
}
#undef TT_STRIP_MMA

__device__ __forceinline__ void cp16(void* dst, const void* src, int bytes) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(s_u32(dst)), "l"(src), "r"(bytes) : "memory");
}
__device__ __forceinline__ void cp4(void* dst, const void* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(s_u32(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// Asynchronous copy of one tile of X (tb rows of i_d, ta entries of i_1 each)
// into the raw buffer (rows of TA + 4 words).  Rows that do not start on 16
// bytes (a.vec = 0) are copied from the 16-byte boundary below, so entry i of
// row r lies at word (start word mod 4) + i; copies never leave the slab.
__device__ __forceinline__ void issue_x(const StripArgs& a, const float* src, int ta, int tb, float* raw) {
  const int total = a.cpr * tb;
  for (int o = threadIdx.x; o < total; o += kThreads) {
    const int r = (int)(((uint32_t)o * a.inv_cpr) >> 20), c = o - r * a.cpr;
    const float* p = src + a.Nd1 * r;
    float* d = raw + r * (a.TA + 4) + 4 * c;
    if (a.vec) {
      if (4 * c < ta) cp16(d, p + 4 * c, min(16, 4 * (ta - 4 * c)));
    } else {
      const float* q = reinterpret_cast<const float*>(reinterpret_cast<uintptr_t>(p) & ~(uintptr_t)15) + 4 * c;
      if (q >= p + ta) continue;
      if (q >= a.X && q + 4 <= a.X + a.total) {
        cp16(d, q, 16);
      } else {
        for (int e = 0; e < 4; ++e)
          if (q + e >= p && q + e < p + ta) cp4(d + e, q + e);
      }
    }
  }
}

template <int FMT>
__device__ __forceinline__ void put_split2(const StripArgs& a, float x0, float x1, char* h, char* l) {
  if constexpr (FMT == kFmtTF32) {
    const float2 hi = make_float2(round_tf32(x0), round_tf32(x1));
    *reinterpret_cast<float2*>(h) = hi;
    *reinterpret_cast<float2*>(l) = make_float2(round_tf32(__fsub_rn(x0, hi.x)), round_tf32(__fsub_rn(x1, hi.y)));
  } else {
    if constexpr (FMT == kFmtFP16) {
      x0 = __fmul_rn(x0, a.xscale);
      x1 = __fmul_rn(x1, a.xscale);
    }
    tc::split_hi_lo<FMT == kFmtFP16>(x0, x1, *reinterpret_cast<uint32_t*>(h), *reinterpret_cast<uint32_t*>(l));
  }
}

// The raw tile into hi and lo parts [b][a]; zero up to TA columns and tbk rows.
// Aligned rows: a thread converts the chunks that it copied itself.
template <int FMT>
__device__ __forceinline__ void convert_x(const StripArgs& a, const float* src, int ta, int tb, int tbk,
                                          const float* raw, char* xh, char* xl) {
  constexpr int E = esz(FMT);
  const int ldb = (a.TA + 8) * E, qpr = a.TA >> 2;
  if (a.vec) {
#pragma unroll 4
    for (int o = threadIdx.x; o < qpr * tbk; o += kThreads) {
      const int r = (int)(((uint32_t)o * a.inv_qpr) >> 20), q = o - r * qpr;
      float4 v = *reinterpret_cast<const float4*>(raw + r * (a.TA + 4) + 4 * q);
      if (r >= tb || 4 * q + 3 >= ta) {
        if (r >= tb || 4 * q >= ta) v.x = 0.f;
        if (r >= tb || 4 * q + 1 >= ta) v.y = 0.f;
        if (r >= tb || 4 * q + 2 >= ta) v.z = 0.f;
        v.w = 0.f;
      }
      const int d = r * ldb + 4 * E * q;
      if constexpr (FMT == kFmtTF32) {
        put_split2<FMT>(a, v.x, v.y, xh + d, xl + d);
        put_split2<FMT>(a, v.z, v.w, xh + d + 8, xl + d + 8);
      } else {
        if constexpr (FMT == kFmtFP16) {
          v.x = __fmul_rn(v.x, a.xscale);
          v.y = __fmul_rn(v.y, a.xscale);
          v.z = __fmul_rn(v.z, a.xscale);
          v.w = __fmul_rn(v.w, a.xscale);
        }
        uint2 h, l;
        tc::split_hi_lo<FMT == kFmtFP16>(v.x, v.y, h.x, l.x);
        tc::split_hi_lo<FMT == kFmtFP16>(v.z, v.w, h.y, l.y);
        *reinterpret_cast<uint2*>(xh + d) = h;
        *reinterpret_cast<uint2*>(xl + d) = l;
      }
    }
  } else {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t sh0 = (uint32_t)(reinterpret_cast<uintptr_t>(src) >> 2), dsh = (uint32_t)a.Nd1;
    for (int r = warp; r < tbk; r += kWarps) {
      const float* p = raw + r * (a.TA + 4) + ((sh0 + dsh * (uint32_t)r) & 3u);
      for (int i = 2 * lane; i < a.TA; i += 64) {
        const float x0 = r < tb && i < ta ? p[i] : 0.f, x1 = r < tb && i + 1 < ta ? p[i + 1] : 0.f;
        put_split2<FMT>(a, x0, x1, xh + r * ldb + E * i, xl + r * ldb + E * i);
      }
    }
  }
}

// One test-matrix quad (four normals or factor products of row r) into the
// staged block.
template <int FMT>
__device__ __forceinline__ void put_quad(char* gs, int ldg, int r, int q, float4 z, int width) {
  const float z0 = 4 * q < width ? z.x : 0.f, z1 = 4 * q + 1 < width ? z.y : 0.f;
  const float z2 = 4 * q + 2 < width ? z.z : 0.f, z3 = 4 * q + 3 < width ? z.w : 0.f;
  char* p = gs + r * ldg + 4 * esz(FMT) * q;
  if constexpr (FMT == kFmtTF32)
    *reinterpret_cast<float4*>(p) = make_float4(round_tf32(z0), round_tf32(z1), round_tf32(z2), round_tf32(z3));
  else
    *reinterpret_cast<uint2*>(p) =
        make_uint2(tc::op16x2_bits<FMT == kFmtFP16>(z0, z1), tc::op16x2_bits<FMT == kFmtFP16>(z2, z3));
}

// Khatri-Rao rows (kept out of line: the dense path then needs no registers
// for it).  Rows grow0 + gstep r; a mode-by-mode sketch takes its mode-1 factor
// rows f0 + r instead.
template <int FMT, int NT>
__device__ __noinline__ void stage_g_kr(const char* wsb, const DevSketch* krs, int mbm, char* gs, int nr, int64_t grow0,
                                        int64_t gstep, int64_t f0, int width) {
  constexpr int NQ = 2 * NT, LDG = ldg_bytes(FMT, NT);
  for (int o = threadIdx.x; o < nr * NQ; o += kThreads) {
    const int r = o / NQ, q = o - r * NQ;
    float4 z = make_float4(0.f, 0.f, 0.f, 0.f);
    if (4 * q < width)
      z = mbm ? kr_f1_quad(wsb, *krs, f0 + r, (uint32_t)q)
              : kr_quad_f32(wsb, *krs, (uint64_t)(grow0 + gstep * r), (uint32_t)q);
    put_quad<FMT>(gs, LDG, r, q, z, width);
  }
}

template <int FMT, int NT>
__device__ __forceinline__ void zero_rows(char* gs, int nr, int kext) {
  constexpr int LDG = ldg_bytes(FMT, NT), NCH = NT * esz(FMT) / 2;
  for (int o = threadIdx.x; o < (kext - nr) * NCH; o += kThreads) {
    const int r = nr + o / NCH, c = o % NCH;
    *reinterpret_cast<uint4*>(gs + r * LDG + 16 * c) = make_uint4(0, 0, 0, 0);
  }
}

// One sketch's test-matrix rows of a tile, rows nr..kext zero: nr rows copied
// (asynchronously) from row trow of its table ...
template <int FMT, int NT>
__device__ __forceinline__ void copy_g(const StripArgs& a, const StSk& s, char* gs, int nr, int kext, int64_t trow) {
  constexpr int E = esz(FMT), LDG = ldg_bytes(FMT, NT);
  constexpr int NCH = NT * E / 2;   // 16-byte chunks of a row
  const int cpr = s.lpad * E / 16;
  const uint4* src = reinterpret_cast<const uint4*>(a.wsb + s.tab) + trow * cpr;
  for (int o = threadIdx.x; o < nr * NCH; o += kThreads) {
    const int r = o / NCH, c = o - r * NCH;
    if (c < cpr) cp16(gs + r * LDG + 16 * c, src + r * cpr + c, 16);
    else *reinterpret_cast<uint4*>(gs + r * LDG + 16 * c) = make_uint4(0, 0, 0, 0);
  }
  zero_rows<FMT, NT>(gs, nr, kext);
}

// ... or generated: rows grow0 + gstep r of the test matrix.
template <int FMT, int NT>
__device__ __forceinline__ void make_g(const StripArgs& a, const StSk& s, char* gs, int nr, int kext, int64_t grow0,
                                       int64_t gstep, int64_t f0) {
  constexpr int LDG = ldg_bytes(FMT, NT);
  if (s.kr >= 0) {
    stage_g_kr<FMT, NT>(a.wsb, ws_sketches(a.wsb) + s.kr, s.mbm, gs, nr, grow0, gstep, f0, s.width);
  } else {
    // two Philox chains per thread at a time
    constexpr int NQ = 2 * NT;
    const int nq = (s.width + 3) >> 2, jobs = nr * NQ;
    for (int o0 = threadIdx.x; o0 < jobs; o0 += 2 * kThreads) {
      float4 z[2];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int o = min(o0 + h * kThreads, jobs - 1);
        const int r = o / NQ, q = o - r * NQ;
        z[h] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (q < nq) z[h] = normals4_f32(a.seed, (uint32_t)s.sid, (uint64_t)(grow0 + gstep * r), (uint32_t)q);
      }
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int o = o0 + h * kThreads;
        if (o < jobs) put_quad<FMT>(gs, LDG, o / NQ, o % NQ, z[h], s.width);
      }
    }
  }
  zero_rows<FMT, NT>(gs, nr, kext);
}

// A fragments (hi and lo) of a 32-deep contraction chunk: KS k-steps of 16
// (16-bit) or 8 (TF32).  COL: M = i_1, K = i_d, the [b][a] tile read
// transposed; else M = i_d, K = i_1, as stored.  Steps at or past kend are
// skipped (their fragments are not used).
template <int FMT, bool COL>
__device__ __forceinline__ void load_a(uint32_t xs, int ldb, int m0, int k0, uint32_t* f) {
  const int lane = threadIdx.x & 31;
  if constexpr (FMT != kFmtTF32) {
    if constexpr (COL)
      ldsm4t(xs + (k0 + (lane & 7) + 8 * (lane >> 4)) * ldb + 2 * (m0 + 8 * ((lane >> 3) & 1)), f);
    else
      ldsm4(xs + (m0 + (lane & 7) + 8 * ((lane >> 3) & 1)) * ldb + 2 * (k0 + 8 * (lane >> 4)), f);
  } else {
    const int g = lane >> 2, t = lane & 3;
    const int sm = COL ? 4 : ldb, sk = COL ? ldb : 4;
    const uint32_t p = xs + (m0 + g) * sm + (k0 + t) * sk;
    f[0] = __float_as_uint(lds_f(p));
    f[1] = __float_as_uint(lds_f(p + 8 * sm));
    f[2] = __float_as_uint(lds_f(p + 4 * sk));
    f[3] = __float_as_uint(lds_f(p + 8 * sm + 4 * sk));
  }
}

// t = X'(m0.., k0..) G(k0.., :) of one k-step (FIRST), or added to t; hi and lo
// parts of X.
template <int FMT, int NT, bool FIRST>
__device__ __forceinline__ void step(float (*t)[4], const uint32_t* xh, const uint32_t* xl, uint32_t gs, int k0) {
  const int lane = threadIdx.x & 31;
  constexpr int LDG = ldg_bytes(FMT, NT);
  if constexpr (FMT != kFmtTF32) {
    const uint32_t p = gs + (k0 + (lane & 7) + 8 * ((lane >> 3) & 1)) * LDG + 16 * (lane >> 4);
    uint32_t b[(NT + 1) / 2][4];
#pragma unroll
    for (int n = 0; n + 1 < NT; n += 2) ldsm4t(p + 16 * n, b[n / 2]);
    if constexpr (NT & 1) ldsm2t(gs + (k0 + (lane & 15)) * LDG + 16 * (NT - 1), b[NT / 2]);
#pragma unroll
    for (int n = 0; n < NT; ++n) mma<FMT, FIRST>(t[n], xh, b[n / 2] + 2 * (n & 1));
#pragma unroll
    for (int n = 0; n < NT; ++n) mma<FMT, false>(t[n], xl, b[n / 2] + 2 * (n & 1));
  } else {
    const int g = lane >> 2, tq = lane & 3;
    const uint32_t p = gs + (k0 + tq) * LDG + 4 * g;
    uint32_t b[NT][2];
#pragma unroll
    for (int n = 0; n < NT; ++n) {
      b[n][0] = __float_as_uint(lds_f(p + 32 * n));
      b[n][1] = __float_as_uint(lds_f(p + 32 * n + 4 * LDG));
    }
#pragma unroll
    for (int n = 0; n < NT; ++n) mma<FMT, FIRST>(t[n], xh, b[n]);
#pragma unroll
    for (int n = 0; n < NT; ++n) mma<FMT, false>(t[n], xl, b[n]);
  }
}

// What one tile needs, worked out once (a lane per sketch) while the tile
// before it is multiplied.
struct TileDesc {
  const float* src;
  int b0, gi;
  uint32_t kL;
  int64_t key[kMaxCol + kMaxRow];    // first staged row of each sketch's block (identifies it)
  int64_t grow[kMaxCol + kMaxRow];   // its first test-matrix row
  uint32_t wlo[kMaxCol + kMaxRow];   // w mod wdiv
};

template <int FMT, int NT, int NCOL>
__global__ void __launch_bounds__(kThreads, NCOL * NT <= 12 ? 2 : 1)
    sketch_strip_kernel(const __grid_constant__ StripArgs a) {
  extern __shared__ __align__(16) char sm[];
  __shared__ TileDesc td[2];
  constexpr int E = esz(FMT), KSTEP = FMT == kFmtTF32 ? 8 : 16, KS = 32 / KSTEP;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int g = lane >> 2, tq = lane & 3;
  const int ldb = (a.TA + 8) * E;
  char* xh = sm;
  char* xl = sm + a.off_xl;
  float* raw = reinterpret_cast<float*>(sm + a.off_raw);
  float4* racc = reinterpret_cast<float4*>(sm + a.off_acc);
  float* scale = reinterpret_cast<float*>(sm + a.off_scale);
  double* ws = reinterpret_cast<double*>(a.wsb);
  const int mtB = a.TB >> 4;

  // ---- this CTA's unit: strip ab of i_1, column tiles [gt0, gt0 + ng), kL
  // positions [u0, u1)
  uint32_t unit = blockIdx.x;
  const int ab = (int)(unit % (uint32_t)a.nA);
  unit /= (uint32_t)a.nA;
  const uint32_t gt0 = (unit % (uint32_t)a.nGS) * (uint32_t)a.NG;
  const uint32_t u0 = (unit / (uint32_t)a.nGS) * a.CL;
  const uint32_t u1 = min(a.WL, u0 + a.CL);
  const int ng = (int)min((uint32_t)a.NG, a.ngt - gt0);
  const int a0 = ab * a.TA;
  const int ta = (int)imin64(a.TA, a.n1 - a0);
  const int tak = (ta + 15) & ~15;
  const int nacc = ng * a.nrow * mtB * NT * 32;   // float4 words of the row sums
  for (int i = tid; i < nacc; i += kThreads) racc[i] = make_float4(0.f, 0.f, 0.f, 0.f);

  // descriptor of (position u, column tile gi), by one warp.  kL of position u:
  // the slower digit (i_2) runs slowest, so that the outer column sketches'
  // rows stay as long as they can
  auto describe = [&](TileDesc& d, uint32_t u, int gi) {
    const uint32_t kL = a.q3 == 1 ? u : u / a.q3 + a.q2 * (u % a.q3);
    const uint32_t gt = gt0 + gi, kR = gt / (uint32_t)a.nB;
    const int b0 = (int)(gt - kR * (uint32_t)a.nB) * a.TB;
    if (lane == 0) {
      d.src = a.X + a0 + a.n1 * ((int64_t)kL + (int64_t)a.WL * kR) + a.Nd1 * (int64_t)b0;
      d.b0 = b0;
      d.gi = gi;
      d.kL = kL;
    }
    if (lane < a.ncol) {
      const StSk& sk = a.col[lane];
      const uint32_t hi = kL / sk.wdiv;
      const int64_t whi = (int64_t)hi + (int64_t)(a.WL / sk.wdiv) * kR;
      d.wlo[lane] = kL - hi * sk.wdiv;
      d.key[lane] = whi * a.cnt + b0;
      d.grow[lane] = whi + sk.hstride * (a.first + b0);
    } else if (lane >= kMaxCol && lane < kMaxCol + a.nrow) {
      const StSk& sk = a.row[lane - kMaxCol];
      const uint32_t q = sk.wdiv / a.WL;
      const uint32_t wlo = kL + a.WL * (kR % q);
      d.wlo[lane] = wlo;
      d.key[lane] = d.grow[lane] = (int64_t)wlo * a.n1 + a0;
    }
  };

  float acc[NCOL][NT][4];
  int64_t ckey[NCOL], rkey[kMaxRow];
  uint32_t cwlo[NCOL];
  int adds[NCOL];
#pragma unroll
  for (int s = 0; s < NCOL; ++s) {
    adds[s] = 0;
    cwlo[s] = 0;
    ckey[s] = -1;
#pragma unroll
    for (int n = 0; n < NT; ++n)
#pragma unroll
      for (int e = 0; e < 4; ++e) acc[s][n][e] = 0.0f;
  }
#pragma unroll
  for (int r = 0; r < kMaxRow; ++r) rkey[r] = -1;

  auto flush_col = [&](int s) {
    // rows a0 + 16 warp + g (+ 8) of i_1, columns 8 n + 2 tq (+ 1)
    const StSk& sk = a.col[s];
    if (16 * warp < ta) {
      double* out = ws + sk.off + a.n1 * (int64_t)cwlo[s] + a0 + 16 * warp + g + sk.rows * (2 * tq);
      const bool i0 = 16 * warp + g < ta, i1 = 16 * warp + g + 8 < ta;
#pragma unroll
      for (int n = 0; n < NT; ++n) {
        const int j = 8 * n + 2 * tq;
        if (j < sk.width) {
          if (i0) atomicAdd(out, (double)acc[s][n][0]);
          if (i1) atomicAdd(out + 8, (double)acc[s][n][2]);
        }
        if (j + 1 < sk.width) {
          if (i0) atomicAdd(out + sk.rows, (double)acc[s][n][1]);
          if (i1) atomicAdd(out + sk.rows + 8, (double)acc[s][n][3]);
        }
        out += 8 * sk.rows;
        acc[s][n][0] = acc[s][n][1] = acc[s][n][2] = acc[s][n][3] = 0.0f;
      }
    }
    adds[s] = 0;
  };
  auto flush_rows = [&]() {
    for (int i = tid; i < nacc; i += kThreads) {
      const float4 v = racc[i];
      racc[i] = make_float4(0.f, 0.f, 0.f, 0.f);
      int q = i >> 5;
      const int n = q % NT;
      q /= NT;
      const int mt = q % mtB;
      q /= mtB;
      const int r = q % a.nrow, gi = q / a.nrow;
      const uint32_t gt = gt0 + gi, kR = gt / (uint32_t)a.nB;
      const int b0 = (int)(gt - kR * (uint32_t)a.nB) * a.TB;
      const StSk& sk = a.row[r];
      const int64_t whi = kR / (sk.wdiv / a.WL);
      const float x[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const int l2 = i & 31;
        const int b = b0 + 16 * mt + (l2 >> 2) + 8 * (e >> 1), j = 8 * n + 2 * (l2 & 3) + (e & 1);
        if (b < a.cnt && j < sk.width && x[e] != 0.0f)
          atomicAdd(ws + sk.off + whi + sk.hstride * (a.first + b) + sk.rows * j, (double)x[e]);
      }
    }
  };

  const uint32_t ntile = (u1 - u0) * (uint32_t)ng;
  if (warp == 0) describe(td[0], u0, 0);
  __syncthreads();
  issue_x(a, td[0].src, ta, (int)imin64(a.TB, a.cnt - td[0].b0), raw);
  cp_commit();
  uint32_t nu = u0;   // the next tile's position and column tile
  int ngi = 0, row_adds = 0;
  const uint32_t xhs = s_u32(xh), xls = s_u32(xl);
  for (uint32_t t = 0; t < ntile; ++t) {
    const TileDesc& d = td[t & 1];
    const int tb = (int)imin64(a.TB, a.cnt - d.b0), tbk = (tb + 15) & ~15;
    if (t) __syncthreads();   // products of the tile before are done
    // ---- test-matrix blocks whose rows changed: copies first (asynchronous),
    // then the tile of X, then the generated ones
    bool cnew[NCOL], rnew[kMaxRow];
#pragma unroll
    for (int s = 0; s < NCOL; ++s) {
      cnew[s] = false;
      if (s < a.ncol) {
        // a column sketch whose rows move on goes out first
        if (d.wlo[s] != cwlo[s] && adds[s]) flush_col(s);
        cwlo[s] = d.wlo[s];
        cnew[s] = d.key[s] != ckey[s];
        ckey[s] = d.key[s];
        const StSk& sk = a.col[s];
        if (cnew[s] && sk.tab >= 0) copy_g<FMT, NT>(a, sk, sm + sk.soff, tb, tbk, ckey[s]);
      }
    }
#pragma unroll
    for (int r = 0; r < kMaxRow; ++r) {
      rnew[r] = false;
      if (r < a.nrow) {
        rnew[r] = d.key[kMaxCol + r] != rkey[r];
        rkey[r] = d.key[kMaxCol + r];
        const StSk& sk = a.row[r];
        if (rnew[r] && sk.tab >= 0) copy_g<FMT, NT>(a, sk, sm + sk.soff, ta, tak, rkey[r]);
      }
    }
    cp_commit();
    cp_wait<1>();             // this thread's copies of the X tile
    if (!a.vec) __syncthreads();
    convert_x<FMT>(a, d.src, ta, tb, tbk, raw, xh, xl);
#pragma unroll
    for (int s = 0; s < NCOL; ++s)
      if (cnew[s] && a.col[s].tab < 0) {
        const StSk& sk = a.col[s];
        make_g<FMT, NT>(a, sk, sm + sk.soff, tb, tbk, d.grow[s], sk.hstride, 0);
      }
#pragma unroll
    for (int r = 0; r < kMaxRow; ++r)
      if (rnew[r] && a.row[r].tab < 0) {
        const StSk& sk = a.row[r];
        make_g<FMT, NT>(a, sk, sm + sk.soff, ta, tak, d.grow[kMaxCol + r], 1, a0);
        if (sk.mbm && tid < 2 * NT) {
          float4 c = make_float4(0.f, 0.f, 0.f, 0.f);
          if (4 * tid < sk.width)
            c = kr_scale_quad(a.wsb, ws_sketches(a.wsb)[sk.kr], (uint64_t)d.wlo[kMaxCol + r], (uint32_t)tid,
                              FMT == kFmtTF32 ? TT_PREC_TF32 : FMT == kFmtFP16 ? TT_PREC_FP16 : TT_PREC_BF16);
          reinterpret_cast<float4*>(scale)[tid] = c;
        }
      }
    if (++ngi == ng) ngi = 0, ++nu;
    if (warp == 0 && t + 1 < ntile) describe(td[(t + 1) & 1], nu, ngi);
    cp_wait<0>();
    __syncthreads();
    if (t + 1 < ntile) {      // the next tile travels while this one is multiplied
      const TileDesc& nd = td[(t + 1) & 1];
      issue_x(a, nd.src, ta, (int)imin64(a.TB, a.cnt - nd.b0), raw);
    }
    cp_commit();
    // ---- column products of this warp's m-tile
    if (16 * warp < ta) {
#pragma unroll 1
      for (int kc = 0; kc < tbk; kc += 32) {
        uint32_t fh[KS][4], fl[KS][4];
        const bool full = kc + 16 < tbk;   // 32 of the contraction, else 16
#pragma unroll
        for (int k = 0; k < KS; ++k)
          if (2 * k < KS || full) {
            load_a<FMT, true>(xhs, ldb, 16 * warp, kc + KSTEP * k, fh[k]);
            load_a<FMT, true>(xls, ldb, 16 * warp, kc + KSTEP * k, fl[k]);
          }
#pragma unroll
        for (int s = 0; s < NCOL; ++s)
          if (s < a.ncol) {
            float v[NT][4];
            const uint32_t gs = s_u32(sm + a.col[s].soff);
            step<FMT, NT, true>(v, fh[0], fl[0], gs, kc);
#pragma unroll
            for (int k = 1; k < KS; ++k)
              if (2 * k < KS || full) step<FMT, NT, false>(v, fh[k], fl[k], gs, kc + KSTEP * k);
#pragma unroll
            for (int n = 0; n < NT; ++n)
#pragma unroll
              for (int e = 0; e < 4; ++e) acc[s][n][e] += v[n][e];
          }
      }
    }
    // ---- row products (m-tile of i_d, sketch) of this warp
#pragma unroll 1
    for (int q = 0; q < kMaxTasks; ++q) {
      const int tk = a.task[warp][q];
      if (tk == 255) break;
      const int mt = tk & 7, r = tk >> 3;
      if (16 * mt >= tb) continue;
      const uint32_t gs = s_u32(sm + a.row[r].soff);
      float v[NT][4];
#pragma unroll
      for (int n = 0; n < NT; ++n) v[n][0] = v[n][1] = v[n][2] = v[n][3] = 0.0f;
#pragma unroll 1
      for (int kc = 0; kc < tak; kc += 32) {
        float w[NT][4];
        const bool full = kc + 16 < tak;
#pragma unroll
        for (int k = 0; k < KS; ++k)
          if (2 * k < KS || full) {
            uint32_t fh[4], fl[4];
            load_a<FMT, false>(xhs, ldb, 16 * mt, kc + KSTEP * k, fh);
            load_a<FMT, false>(xls, ldb, 16 * mt, kc + KSTEP * k, fl);
            if (k == 0) step<FMT, NT, true>(w, fh, fl, gs, kc);
            else step<FMT, NT, false>(w, fh, fl, gs, kc + KSTEP * k);
          }
#pragma unroll
        for (int n = 0; n < NT; ++n)
#pragma unroll
          for (int e = 0; e < 4; ++e) v[n][e] += w[n][e];
      }
      float4* p = racc + ((d.gi * a.nrow + r) * mtB + mt) * NT * 32 + lane;
      const bool mbm = a.row[r].mbm != 0;
#pragma unroll
      for (int n = 0; n < NT; ++n) {
        float c0 = 1.0f, c1 = 1.0f;
        if (mbm) c0 = scale[8 * n + 2 * tq], c1 = scale[8 * n + 2 * tq + 1];
        float4 w = p[32 * n];
        w.x += v[n][0] * c0;
        w.y += v[n][1] * c1;
        w.z += v[n][2] * c0;
        w.w += v[n][3] * c1;
        p[32 * n] = w;
      }
    }
    // FP32 sums are bounded; the rest of the summation is FP64
    const int ch = (tbk + 31) >> 5;
#pragma unroll
    for (int s = 0; s < NCOL; ++s)
      if (s < a.ncol) {
        adds[s] += ch;
        if (adds[s] + ch > kAddsMax) flush_col(s);
      }
    if (d.gi == ng - 1 && ++row_adds == kRowAddsMax) {
      row_adds = 0;
      __syncthreads();
      flush_rows();
    }
  }
#pragma unroll
  for (int s = 0; s < NCOL; ++s)
    if (s < a.ncol && adds[s]) flush_col(s);
  __syncthreads();
  if (row_adds) flush_rows();
}

using KernelFn = void (*)(const StripArgs);
// The instances of one format: column octets NT (smallest compiled one that
// holds nt) and NCOL = 2 or 3 column-sketch slots.
KernelFn kernel_bf16(int nt, int ncol);
KernelFn kernel_tf32(int nt, int ncol);
KernelFn kernel_fp16(int nt, int ncol);
template <int FMT>
KernelFn kernel_of(int nt, int ncol) {
  if (ncol <= 2) {
    switch (nt) {
      case 2: return sketch_strip_kernel<FMT, 2, 2>;
      case 3: return sketch_strip_kernel<FMT, 3, 2>;
      case 4: return sketch_strip_kernel<FMT, 4, 2>;
      case 5: return sketch_strip_kernel<FMT, 5, 2>;
      case 6: return sketch_strip_kernel<FMT, 6, 2>;
      default: return sketch_strip_kernel<FMT, 8, 2>;
    }
  }
  switch (nt) {
    case 2: return sketch_strip_kernel<FMT, 2, 3>;
    case 3: return sketch_strip_kernel<FMT, 3, 3>;
    case 4: return sketch_strip_kernel<FMT, 4, 3>;
    case 5: return sketch_strip_kernel<FMT, 5, 3>;
    case 6: return sketch_strip_kernel<FMT, 6, 3>;
    default: return sketch_strip_kernel<FMT, 8, 3>;
  }
}

}  // namespace strip
}  // namespace tts
