// Strip kernel: launch arguments and the device code of one operand format;
// sketch_strip_<format>.cu instantiate it, sketch_strip.cu plans the launch.
//
// The fused multi-sketch (BF16, FP16 or TF32 tensor cores, X split into hi +
// lo) for the shapes that the tcgen05 kernels do not take, with one to three sketches
// a side (of small planes, n_1 and n_d <= 32: dense test matrices).  See sketch_strip.cu
// for the split of the work.
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
constexpr int kDescWarp = kWarps - 1;     // describes the tiles, two ahead: the warp with the fewest column rows
// What that costs, in row-product columns (planning): 200 changed nothing at 960^3, 24^6, 96^4 x 48 and
// 61 x 53 x 67 x 47, so it only has to be of a row product's size.
constexpr int kDescLoad = 96;
constexpr int kWarpTasks = 4;             // row products (m-tile, sketch) of one warp and tile, at most
// FP32 additions into one register accumulator between FP64 flushes: 12 leave the column sums
// closer than the 64 x 32 tile kernel's, which went to FP64 after each 32 terms (BF16, 112 x 100 x
// 100 x 112: 1.002e-7 against 1.005e-7; 32 additions 1.26e-7, 16 1.02e-7, 8 0.93e-7).  96^4 x 48, l = 28: 54.1
// ms with 32, 54.9 with 16, 56.5 with 8, 61.6 with 4.
constexpr int kAddsMax = 12;
constexpr int kRowAddsMax = 16;           // the same for the row sketches' shared sums (4 chunks each)
constexpr int kFmtBF16 = 0, kFmtTF32 = 1, kFmtFP16 = 2;

__host__ __device__ constexpr int esz(int fmt) { return fmt == kFmtTF32 ? 4 : 2; }
__host__ __device__ constexpr int ldg_bytes(int fmt, int nt) { return strip_row_bytes(fmt == kFmtTF32, nt); }

struct StSk {
  int64_t rows, off, hstride;
  int64_t tab;          // byte offset (from the workspace base) of the staged rows, -1: generated
  uint32_t wdiv;        // N_k / n_1
  int width, nq, sid;   // nq: column quads
  int kr;               // global sketch index when the test matrix is Khatri-Rao, -1: dense
  int mbm;              // mode-by-mode Khatri-Rao sketch (scaled per plane)
  int soff;             // byte offset of its staged block(s) in shared memory
  int per;              // a block per grouped plane index (S_1: kL, R_{d-1}: kR), else one
  // How the rows follow from the digits (no division in the tile loop).  Column
  // sketch: w mod wdiv = 0, i_2 or kL and kL div wdiv = kL, i_3 or 0 (kind 0, 1, 2).
  // Row sketch: kR mod (wdiv / WL) = 0, r_lo or kR and the quotient kR, r_hi or 0.
  int kind;
  int64_t mulr;         // column sketch: WL / wdiv
  float inv_nq;         // 1 / nq
  int rpi;              // rows a pass of the block generates: kThreads / nq
};

struct StripArgs {
  const float* X;
  char* wsb;
  int item;                   // index in its plan (batched launches)
  int64_t n1, cnt, first, Nd1;
  uint64_t seed;
  PhiloxKeys keys;            // of the seed
  uint32_t WL, WR, q2, q3;    // kL = i_2 + q2 i_3 (q2 q3 = WL)
  int ncol, nrow, vec;
  uint32_t tabs;              // bit s (columns), kMaxCol + r (rows): the sketch has a table
  float xscale;
  int nA, TA, nB, TB;         // strips of i_1 and tiles of i_d; a tile is TA x TB with its padding
  // Grouped planes (small n_1, n_d): a tile holds PL consecutive i_2 (n1p columns
  // each) and PR values of i_{d-1} (ndp rows each); PL, PR > 1 only with one strip
  // or one tile of the plane.  kR = r_lo + sR r_hi, r_hi = i_{d-1} < nrh.
  int PL, PR, n1p, ndp;
  uint32_t sR, nrh;
  uint32_t npos;              // positions u: groups of i_2 times i_3
  uint32_t ngt;               // column tiles (r_lo, group of r_hi, i_d block)
  int NG, nGS;                // column tiles per unit, sets of them
  uint32_t CL;                // positions per unit
  int cpr;                    // 16-byte chunks copied per row (unaligned rows: one more)
  int rawld;                  // words of a raw row
  float inv_pl;               // 1 / PL
  int off_xl, off_raw, off_g, off_acc, off_scale;   // shared-memory byte offsets
  int64_t total;              // entries of the slab (bounds of the 16-byte copies)
  StSk col[kMaxCol], row[kMaxRow];
  uint8_t task[kWarps][kWarpTasks];  // row products of each warp: m-tile + 8 sketch, 255: none
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

// floor(n / d) of small non-negative integers (n d < 2^22) from inv = 1 / d.
__device__ __forceinline__ int fdiv(int n, float inv) { return (int)(((float)n + 0.5f) * inv); }

// What one tile needs, worked out once (a lane per sketch) while the tile
// before it is multiplied.
struct TileDesc {
  int64_t base;            // entry of the slab at (i_1 = a0, first plane, first i_d)
  int b0, gi;
  int nl, nr, ta, tb;      // planes along kL and kR, valid i_1 and i_d of each
  float inv_ta, inv_tb;
  int64_t key[kMaxCol + kMaxRow];    // first staged row of each sketch's block (identifies it)
  int64_t grow[kMaxCol + kMaxRow];   // its first test-matrix row
  uint32_t wlo[kMaxCol + kMaxRow];   // w mod wdiv of the first plane
  uint32_t fresh;                    // bit s: sketch s's block must be staged (its rows changed)
  uint32_t flush;                    // bit s: column sketch s's sums go out before this tile ...
  uint32_t fwlo[kMaxCol];            // ... to the rows of this w mod wdiv
};

// Per CTA and unit: the cursor over the tiles (kDescWarp's) and every warp's row products.
struct UnitState {
  uint32_t i2, i3, rg, rlo;
  int bb, gi, adds[kMaxCol];
  struct {
    uint32_t gs;   // its test-matrix block in shared memory
    int acc, mt;   // row-sum offset; m-tile, plane row << 8, mode-by-mode << 16
  } task[kWarps][kWarpTasks];
  int ntask[kWarps];
};
struct LaneMap {   // chunk (four words) and first item of this lane, items per warp
  int v;
  __device__ __forceinline__ void set(int n, int lane) { v = (lane % n) | ((lane / n) << 8) | ((32 / n) << 16); }
  __device__ __forceinline__ int c() const { return v & 255; }
  __device__ __forceinline__ int i0() const { return (v >> 8) & 255; }
  __device__ __forceinline__ int np() const { return v >> 16; }
};
// Asynchronous copies of one tile of X into the raw buffer: row (q, b) holds the
// entries of plane row q at i_d = b0 + b, nl runs of n_1 (consecutive kL: one
// contiguous run).  Rows that do not start on 16 bytes (a.vec = 0) are copied from
// the 16-byte boundary below, so entry i of a row lies at word (start word mod 4) +
// i; no copy leaves the slab.  (One bulk copy per row, 256 to 512 bytes each, was
// slower: 960^3 5.2 ms against 3.4.)
__device__ __forceinline__ void issue_x(const StripArgs& a, const TileDesc& d, float* raw, const LaneMap& m) {
  const int run = a.PL > 1 ? d.nl * (int)a.n1 : d.ta, nrow = d.nr * d.tb;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (a.vec) {
    if (m.i0() >= m.np() || 4 * m.c() >= run) return;   // run <= 128
    const float* base = a.X + d.base + 4 * m.c();
    float* dst = raw + 4 * m.c();
    for (int r = warp * m.np() + m.i0(); r < nrow; r += kWarps * m.np()) {
      const int q = a.PR > 1 ? fdiv(r, d.inv_tb) : 0, b = r - q * d.tb;
      cp16(dst + r * a.rawld, base + a.n1 * ((int64_t)q * a.sR * a.WL) + a.Nd1 * b, 16);
    }
    return;
  }
  for (int r = warp; r < nrow; r += kWarps) {
    const int q = a.PR > 1 ? fdiv(r, d.inv_tb) : 0, b = r - q * d.tb;
    const float* p = a.X + d.base + a.n1 * ((int64_t)q * a.sR * a.WL) + a.Nd1 * b;
    for (int c = lane; c < a.cpr; c += 32) {
      float* dst = raw + r * a.rawld + 4 * c;
      const float* s = reinterpret_cast<const float*>(reinterpret_cast<uintptr_t>(p) & ~(uintptr_t)15) + 4 * c;
      if (s >= p + run) break;
      if (s >= a.X && s + 4 <= a.X + a.total) {
        cp16(dst, s, 16);
      } else {
        for (int e = 0; e < 4; ++e)
          if (s + e >= p && s + e < p + run) cp4(dst + e, s + e);
      }
    }
  }
}

__device__ __forceinline__ void put_split2_tf32(float x0, float x1, char* h, char* l) {
  const float2 hi = make_float2(round_tf32(x0), round_tf32(x1));
  *reinterpret_cast<float2*>(h) = hi;
  *reinterpret_cast<float2*>(l) = make_float2(round_tf32(__fsub_rn(x0, hi.x)), round_tf32(__fsub_rn(x1, hi.y)));
}

// The raw tile into hi and lo parts [b][a].  Everything inside the valid planes'
// padding is zero (set once at the start); planes and rows that this tile lacks are
// written as zeros, since another tile may have had them.
template <int FMT>
__device__ __forceinline__ void convert_x(const StripArgs& a, const TileDesc& d, int tbk, const float* raw, char* xh,
                                          char* xl, const LaneMap& m) {
  constexpr int E = esz(FMT);
  const int ldb = (a.TA + 8) * E, warp = threadIdx.x >> 5;
  const int nbr = a.PR > 1 ? (int)a.cnt : tbk;      // rows written per plane row
  const uint32_t dsh = (uint32_t)a.Nd1, gsh = (uint32_t)(a.n1 * (int64_t)a.sR * a.WL);
  const uint32_t sh0 = a.vec ? 0u : (uint32_t)(reinterpret_cast<uintptr_t>(a.X + d.base) >> 2);
  const int q0 = m.c();   // this lane's column quad of a plane
  if (m.i0() < m.np()) {
    for (int it = warp * m.np() + m.i0(); it < a.PR * nbr * a.PL; it += kWarps * m.np()) {   // (row, plane)
      const int r = a.PL > 1 ? fdiv(it, a.inv_pl) : it, p = it - r * a.PL;
      const int q = a.PR > 1 ? fdiv(r, d.inv_tb) : 0, b = r - q * nbr;
      const bool row_on = q < d.nr && b < d.tb;
      const float* src =
          raw + (q * d.tb + b) * a.rawld + (a.vec ? 0u : ((sh0 + gsh * (uint32_t)q + dsh * (uint32_t)b) & 3u));
      const int drow = (q * a.ndp + b) * ldb;
      {
        const int valid = row_on && p < d.nl ? d.ta : 0;   // entries of this plane's row
        const float* x = src + p * (int)a.n1 + 4 * q0;
        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
        if (a.vec && 4 * q0 + 3 < valid) {
          v = *reinterpret_cast<const float4*>(x);
        } else {
          if (4 * q0 < valid) v.x = x[0];
          if (4 * q0 + 1 < valid) v.y = x[1];
          if (4 * q0 + 2 < valid) v.z = x[2];
          if (4 * q0 + 3 < valid) v.w = x[3];
        }
        const int o = drow + E * (p * a.n1p + 4 * q0);
        if constexpr (FMT == kFmtTF32) {
          put_split2_tf32(v.x, v.y, xh + o, xl + o);
          put_split2_tf32(v.z, v.w, xh + o + 8, xl + o + 8);
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
          *reinterpret_cast<uint2*>(xh + o) = h;
          *reinterpret_cast<uint2*>(xl + o) = l;
        }
      }
    }
  }
}

// One test-matrix quad (four normals or factor products of row r) into the
// staged block.
template <int FMT>
__device__ __forceinline__ void put_quad(char* gs, int ldg, int r, int q, float4 z, int width) {
  float z0 = z.x, z1 = z.y, z2 = z.z, z3 = z.w;
  if (width & 3) {   // uniform: a last quad that is not full
    z1 = 4 * q + 1 < width ? z1 : 0.f;
    z2 = 4 * q + 2 < width ? z2 : 0.f;
    z3 = 4 * q + 3 < width ? z3 : 0.f;
  }
  if constexpr (FMT == kFmtTF32)
    *reinterpret_cast<float4*>(gs + r * ldg + 16 * q) = make_float4(round_tf32(z0), round_tf32(z1), round_tf32(z2), round_tf32(z3));
  else
    *reinterpret_cast<uint2*>(gs + r * ldg + 16 * ((q >> 1) ^ strip_swizzle(ldg / 16, r)) + 8 * (q & 1)) =
        make_uint2(tc::op16x2_bits<FMT == kFmtFP16>(z0, z1), tc::op16x2_bits<FMT == kFmtFP16>(z2, z3));
}

// Rows of one sketch's staged block: blk blocks of (no x ni) rows, row (p, o, i) at
// block row o pad + i of block p (bstep block rows apart), test-matrix row grow + p gp +
// o go + i gi.
struct Rows {
  int nblk, bstep, no, ni, pad;
  int64_t gp, go, gi;
  float inv_ni;
};

// Khatri-Rao rows (kept out of line: the dense path then needs no registers
// for it).  A mode-by-mode sketch takes its mode-1 factor rows f0 + i instead.
template <int FMT, int NT>
__device__ __noinline__ void stage_g_kr(const char* wsb, const DevSketch* krs, int mbm, char* gs, Rows w, int64_t grow,
                                        int64_t f0, int width) {
  constexpr int NQ = 2 * NT, LDG = ldg_bytes(FMT, NT);
  for (int o = threadIdx.x; o < w.no * w.ni * NQ; o += kThreads) {
    const int e = o / NQ, q = o - e * NQ, oo = e / w.ni, i = e - oo * w.ni;
    float4 z = make_float4(0.f, 0.f, 0.f, 0.f);
    if (4 * q < width)
      z = mbm ? kr_f1_quad(wsb, *krs, f0 + i, (uint32_t)q)
              : kr_quad_f32(wsb, *krs, (uint64_t)(grow + w.go * oo + w.gi * i), (uint32_t)q);
    put_quad<FMT>(gs, LDG, oo * w.pad + i, q, z, width);
  }
}

// Generated test-matrix rows.  A thread keeps its quad q and goes through the rows in
// steps of kThreads / nq: no division a quad (KEYS: the Philox keys are launch arguments
// in the constant bank; a batched launch's lie in shared memory and are not used).
template <int FMT, int NT, bool KEYS>
__device__ __forceinline__ void make_g(const StripArgs& a, const StSk& s, char* gs, const Rows& w, int64_t grow,
                                       int64_t f0) {
  constexpr int LDG = ldg_bytes(FMT, NT);
  if (s.kr >= 0) {
    stage_g_kr<FMT, NT>(a.wsb, ws_sketches(a.wsb) + s.kr, s.mbm, gs, w, grow, f0, s.width);
    return;
  }
  const int rows = w.no * w.ni;
  const float inv_rows = __frcp_rn((float)rows);
  const int r0 = fdiv((int)threadIdx.x, s.inv_nq), q = (int)threadIdx.x - r0 * s.nq;
  if (r0 >= s.rpi) return;
  for (int r = r0; r < w.nblk * rows; r += s.rpi) {
    int e = r, p = 0, oo = 0;
    if (w.nblk > 1) p = fdiv(e, inv_rows), e -= p * rows;
    if (w.no > 1) oo = fdiv(e, w.inv_ni), e -= oo * w.ni;
    const uint64_t row = (uint64_t)(grow + w.gp * p + w.go * oo + w.gi * e);
    float4 z;
    if constexpr (KEYS) z = normals4_f32(a.keys, (uint32_t)s.sid, row, (uint32_t)q);
    else z = normals4_f32(a.seed, (uint32_t)s.sid, row, (uint32_t)q);
    put_quad<FMT>(gs, LDG, p * w.bstep + oo * w.pad + e, q, z, s.width);
  }
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

// t = X'(m0.., k0..) G(k0.., :) of one k-step (FIRST), or added to t; lo and hi
// parts of X, the low one first: a tensor-core addition loses up to a unit of the last
// place of its result, and there the result is still small (sums 1.05e-7 off with the high
// part first, 0.87e-7 so; TF32 2.0e-7, 1.7e-7).
template <int FMT, int NT, bool FIRST>
__device__ __forceinline__ void step(float (*t)[4], const uint32_t* xh, const uint32_t* xl, uint32_t gs, int k0) {
  const int lane = threadIdx.x & 31;
  constexpr int LDG = ldg_bytes(FMT, NT);
  if constexpr (FMT != kFmtTF32) {
    // chunk n + (lane >> 4) of row k0 + ..., swizzled: n even, so n + m = n ^ m
    const uint32_t m = (uint32_t)((lane >> 4) ^ strip_swizzle(NT, lane & 7));
    const uint32_t p = gs + (k0 + (lane & 7) + 8 * ((lane >> 3) & 1)) * LDG;
    uint32_t b[(NT + 1) / 2][4];
#pragma unroll
    for (int n = 0; n + 1 < NT; n += 2) ldsm4t(p + 16 * (m ^ (uint32_t)n), b[n / 2]);
    if constexpr (NT & 1) ldsm2t(gs + (k0 + (lane & 15)) * LDG + 16 * (NT - 1), b[NT / 2]);
#pragma unroll
    for (int n = 0; n < NT; ++n) mma<FMT, FIRST>(t[n], xl, b[n / 2] + 2 * (n & 1));
#pragma unroll
    for (int n = 0; n < NT; ++n) mma<FMT, false>(t[n], xh, b[n / 2] + 2 * (n & 1));
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
    for (int n = 0; n < NT; ++n) mma<FMT, FIRST>(t[n], xl, b[n]);
#pragma unroll
    for (int n = 0; n < NT; ++n) mma<FMT, false>(t[n], xh, b[n]);
  }
}

// One unit of work: strip ab of i_1, a set of column tiles, a range of positions.
template <int FMT, int NT, int NCOL, bool KEYS>
__device__ __forceinline__ void strip_unit(const StripArgs& a, uint32_t unit, char* sm, TileDesc* td, UnitState& us, uint64_t* bar,
                                           volatile int* abort_flag) {
  constexpr int E = esz(FMT), KSTEP = FMT == kFmtTF32 ? 8 : 16, KS = 32 / KSTEP, LDG = ldg_bytes(FMT, NT);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int g = lane >> 2, tq = lane & 3;
  const int ldb = (a.TA + 8) * E;
  char* xh = sm;
  char* xl = sm + a.off_xl;
  float* raw = reinterpret_cast<float*>(sm + a.off_raw);
  float4* racc = reinterpret_cast<float4*>(sm + a.off_acc);
  float* scale = reinterpret_cast<float*>(sm + a.off_scale);
  double* ws = reinterpret_cast<double*>(a.wsb);
  int* status = reinterpret_cast<int*>(a.wsb + kStatusOff);
  const int mtB = a.TB >> 4;
  const uint32_t bar_g = s_u32(bar);

  const int ab = (int)(unit % (uint32_t)a.nA);
  unit /= (uint32_t)a.nA;
  const uint32_t gt0 = (unit % (uint32_t)a.nGS) * (uint32_t)a.NG;
  const uint32_t u0 = (unit / (uint32_t)a.nGS) * a.CL;
  const uint32_t u1 = min(a.npos, u0 + a.CL);
  const int ng = (int)min((uint32_t)a.NG, a.ngt - gt0);
  const int a0 = ab * a.TA;
  const int ta = a.PL > 1 ? (int)a.n1 : (int)imin64(a.TA, a.n1 - a0);   // valid i_1 of a plane
  const int tak = a.PL > 1 ? a.TA : (ta + 15) & ~15;
  const int nacc = ng * a.nrow * mtB * NT * 32;   // float4 words of the row sums
  for (int i = tid; i < nacc; i += kThreads) racc[i] = make_float4(0.f, 0.f, 0.f, 0.f);
  // padding of the tile and of the test-matrix blocks: zero, never written again
  for (int i = tid; i < a.off_raw / 16; i += kThreads) reinterpret_cast<uint4*>(sm)[i] = make_uint4(0, 0, 0, 0);
  for (int i = a.off_g / 16 + tid; i < a.off_scale / 16; i += kThreads)
    reinterpret_cast<uint4*>(sm)[i] = make_uint4(0, 0, 0, 0);
  // this warp's m-tile of the strip: plane mp of the group, i_1 from ma on
  const int mp = 16 * warp / a.n1p, ma = 16 * warp - mp * a.n1p;

  // Cursor over the tiles (position slowest): position (i2, i3), column tile gi =
  // (r_lo, rg, bb).  The slower digit i_2 runs slowest, so that the outer column
  // sketches' rows stay as long as they can.
  auto start = [&]() {
    const uint32_t grp = gt0 / (uint32_t)a.nB;
    us.rg = grp / a.sR;
    us.rlo = grp - us.rg * a.sR;
    us.bb = (int)(gt0 - grp * (uint32_t)a.nB);
    us.gi = 0;
  };
  auto advance = [&]() {
    if (us.gi + 1 == ng) {
      start();
      if (us.i3 + 1 == a.q3) us.i3 = 0, us.i2 += (uint32_t)a.PL;
      else ++us.i3;
    } else {
      ++us.gi;
      if (us.bb + 1 == a.nB) {
        us.bb = 0;
        if (us.rlo + 1 == a.sR) us.rlo = 0, ++us.rg;
        else ++us.rlo;
      } else {
        ++us.bb;
      }
    }
  };
  // descriptor of the tile at the cursor, by one warp (a lane per sketch)
  auto describe = [&](TileDesc& d, const TileDesc* prev) {
    const uint32_t i2 = us.i2, i3 = us.i3, rlo = us.rlo;
    const uint32_t kL = i2 + a.q2 * i3, rh = us.rg * (uint32_t)a.PR, kR = rlo + a.sR * rh;
    const int b0 = us.bb * a.TB, tb = (int)imin64(a.PR > 1 ? a.cnt : a.TB, a.cnt - b0);
    if (lane == 0) {
      d.base = a0 + a.n1 * ((int64_t)kL + (int64_t)a.WL * kR) + a.Nd1 * (int64_t)b0;
      d.b0 = b0;
      d.gi = us.gi;
      d.nl = (int)min((uint32_t)a.PL, a.q2 - i2);
      d.nr = (int)min((uint32_t)a.PR, a.nrh - rh);
      d.ta = ta;
      d.tb = tb;
      d.inv_ta = __frcp_rn((float)ta);
      d.inv_tb = __frcp_rn((float)tb);
    }
    bool fresh = false, flush = false;
    if (lane < a.ncol) {
      const StSk& sk = a.col[lane];
      const uint32_t hi = sk.kind == 0 ? kL : sk.kind == 1 ? i3 : 0u;
      const int64_t whi = (int64_t)hi + sk.mulr * kR, key = whi * a.cnt + b0;
      const uint32_t wlo = sk.kind == 0 ? 0u : sk.kind == 1 ? i2 : kL;
      d.wlo[lane] = wlo;
      d.key[lane] = key;
      d.grow[lane] = whi + sk.hstride * (a.first + b0);
      fresh = !prev || prev->key[lane] != key;
      // FP32 sums are bounded; the rest of the summation is FP64
      const int ch = ((a.PR > 1 ? a.TB : tb) + 31) >> 5;
      flush = prev && (prev->wlo[lane] != wlo || us.adds[lane] + ch > kAddsMax);
      us.adds[lane] = flush || !prev ? ch : us.adds[lane] + ch;
      d.fwlo[lane] = prev ? prev->wlo[lane] : 0u;
    } else if (lane >= kMaxCol && lane < kMaxCol + a.nrow) {
      const StSk& sk = a.row[lane - kMaxCol];
      const uint32_t wlo = kL + a.WL * (sk.kind == 0 ? 0u : sk.kind == 1 ? rlo : kR);
      const int64_t key = (int64_t)wlo * a.n1 + a0;
      d.wlo[lane] = wlo;
      d.key[lane] = d.grow[lane] = key;
      fresh = !prev || prev->key[lane] != key;
    }
    const uint32_t bf = __ballot_sync(0xffffffffu, fresh), bl = __ballot_sync(0xffffffffu, flush);
    if (lane == 0) d.fresh = bf, d.flush = bl;
  };

  float acc[NCOL][NT][4];
#pragma unroll
  for (int s = 0; s < NCOL; ++s)
#pragma unroll
    for (int n = 0; n < NT; ++n)
#pragma unroll
      for (int e = 0; e < 4; ++e) acc[s][n][e] = 0.0f;

  auto flush_col = [&](int s, uint32_t w0) {
    // rows (kL + mp, i_1 = a0 + ma + g (+ 8)), columns 8 n + 2 tq (+ 1).  A plane that
    // the group lacks has zero sums: it adds nothing.
    const StSk& sk = a.col[s];
    if (16 * warp < tak) {
      const uint32_t wl = sk.wdiv == 1 ? 0u : w0 + (uint32_t)mp;
      double* out = ws + sk.off + a.n1 * (int64_t)wl + a0 + ma + g + sk.rows * (2 * tq);
      const bool in = a.PL == 1 || sk.wdiv == 1 || wl % a.q2 >= (uint32_t)mp;
      const bool i0 = in && ma + g < ta, i1 = in && ma + g + 8 < ta;
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
      const uint32_t gt = gt0 + gi, grp = gt / (uint32_t)a.nB;
      const int b0 = (int)(gt - grp * (uint32_t)a.nB) * a.TB;
      const int qp = 16 * mt / a.ndp, bm = 16 * mt - qp * a.ndp;   // plane row, first i_d of the m-tile
      const uint32_t rg = grp / a.sR, rh = rg * (uint32_t)a.PR + (uint32_t)qp;
      if (rh >= a.nrh) continue;
      const uint32_t kR = grp - rg * a.sR + a.sR * rh;
      const StSk& sk = a.row[r];
      const int64_t whi = kR / (sk.wdiv / a.WL);
      const float x[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const int l2 = i & 31;
        const int bb = bm + (l2 >> 2) + 8 * (e >> 1), j = 8 * n + 2 * (l2 & 3) + (e & 1);
        if (b0 + bb < a.cnt && j < sk.width && x[e] != 0.0f)
          atomicAdd(ws + sk.off + whi + sk.hstride * (a.first + b0 + bb) + sk.rows * j, (double)x[e]);
      }
    }
  };

  const uint32_t ntile = (u1 - u0) * (uint32_t)ng;
  // lanes of a warp over (chunk of four words, item)
  LaneMap mi, mc;
  mi.set(max(1, (a.PL > 1 ? a.PL * (int)a.n1 : ta) >> 2), lane);   // copies of aligned rows: item = row
  mc.set(((a.PL > 1 ? (int)a.n1 : a.TA) + 3) >> 2, lane);          // conversion: item = (row, plane)
  if (lane < kWarpTasks) {
    const int tk = a.task[warp][lane];
    if (tk != 255) {
      const int mt = tk & 7, r = tk >> 3, qp = 16 * mt / a.ndp;
      us.task[warp][lane].gs = s_u32(sm + a.row[r].soff) + (a.row[r].per ? qp * a.TA * LDG : 0);
      us.task[warp][lane].acc = (r * mtB + mt) * NT * 32;
      us.task[warp][lane].mt = mt | (qp << 8) | (a.row[r].mbm ? 1 << 16 : 0);
    }
    const uint32_t on = __ballot_sync((1u << kWarpTasks) - 1u, tk != 255);
    if (lane == 0) us.ntask[warp] = __popc(on);
  }
  if (warp == kDescWarp) {
    if (lane == 0) {
      us.i2 = u0 / a.q3;
      us.i3 = u0 - us.i2 * a.q3;
      us.i2 *= (uint32_t)a.PL;
      start();
    }
    __syncwarp();
    describe(td[0], nullptr);
    if (ntile > 1) {
      if (lane == 0) advance();
      __syncwarp();
      describe(td[1], &td[0]);
    }
  }
  __syncthreads();
  issue_x(a, td[0], raw, mi);
  cp_commit();
  int row_adds = 0;
  uint32_t gphase = 0;
  const uint32_t xhs = s_u32(xh), xls = s_u32(xl);
  int cur = 0;
  for (uint32_t t = 0; t < ntile; ++t) {
    const TileDesc& d = td[cur];
    const int nxt = cur == 2 ? 0 : cur + 1;
    const int tbk = a.PR > 1 ? a.TB : (d.tb + 15) & ~15;
    cp_wait<0>();
    __syncthreads();          // the raw tile is there; products of the tile before are done
    // ---- test-matrix blocks whose rows changed: tables first (bulk copies by
    // one thread), then the tile of X, then the generated ones
    const uint32_t fresh = d.fresh;
    const bool copies = (fresh & a.tabs) != 0;
#pragma unroll
    for (int s = 0; s < NCOL; ++s)   // a column sketch whose rows move on goes out first
      if (d.flush >> s & 1) flush_col(s, d.fwlo[s]);
    if (copies && tid == 0) {
      uint32_t bytes = 0;
#pragma unroll
      for (int s = 0; s < NCOL; ++s)
        if (fresh & a.tabs & (1u << s)) bytes += (uint32_t)(d.nr * d.tb * LDG);
#pragma unroll
      for (int r = 0; r < kMaxRow; ++r)
        if (fresh & a.tabs & (1u << (kMaxCol + r))) bytes += (uint32_t)((a.row[r].per ? d.nr : 1) * d.nl * d.ta * LDG);
      tc::fence_async_smem();   // the blocks were read (and zeroed) by ordinary accesses
      tc::mbar_arrive_expect_tx(bar_g, bytes);
#pragma unroll
      for (int s = 0; s < NCOL; ++s)
        if (fresh & a.tabs & (1u << s)) {
          const StSk& sk = a.col[s];
          const int64_t dq = sk.mulr * a.sR * a.cnt;
          for (int q = 0; q < d.nr; ++q)
            tc::bulk_g2s(s_u32(sm + sk.soff + q * a.ndp * LDG), a.wsb + sk.tab + (d.key[s] + q * dq) * LDG,
                         (uint32_t)(d.tb * LDG), bar_g);
        }
#pragma unroll
      for (int r = 0; r < kMaxRow; ++r)
        if (fresh & a.tabs & (1u << (kMaxCol + r))) {
          const StSk& sk = a.row[r];
          for (int q = 0; q < (sk.per ? d.nr : 1); ++q)
            for (int p = 0; p < d.nl; ++p)
              tc::bulk_g2s(s_u32(sm + sk.soff + (q * a.TA + p * a.n1p) * LDG),
                           a.wsb + sk.tab + (d.key[kMaxCol + r] + (int64_t)q * a.WL * a.sR * a.n1 + p * a.n1) * LDG,
                           (uint32_t)(d.ta * LDG), bar_g);
        }
    }
    convert_x<FMT>(a, d, tbk, raw, xh, xl, mc);
#pragma unroll
    for (int s = 0; s < NCOL; ++s)
      if (fresh & ~a.tabs & (1u << s)) {
        const StSk& sk = a.col[s];
        const int64_t dq = sk.mulr * a.sR;
        make_g<FMT, NT, KEYS>(a, sk, sm + sk.soff,
                              Rows{sk.per ? d.nl : 1, a.TB, d.nr, d.tb, a.ndp, 1, dq, sk.hstride, d.inv_tb},
                        d.grow[s], 0);
      }
#pragma unroll
    for (int r = 0; r < kMaxRow; ++r)
      if (fresh & ~a.tabs & (1u << (kMaxCol + r))) {
        const StSk& sk = a.row[r];
        make_g<FMT, NT, KEYS>(a, sk, sm + sk.soff,
                        Rows{sk.per ? d.nr : 1, a.TA, d.nl, d.ta, a.n1p, (int64_t)a.WL * a.sR * a.n1, a.n1, 1,
                             d.inv_ta},
                        d.grow[kMaxCol + r], a0);
        if (sk.mbm && tid < 2 * NT) {
          float4 c = make_float4(0.f, 0.f, 0.f, 0.f);
          if (4 * tid < sk.width)
            c = kr_scale_quad(a.wsb, ws_sketches(a.wsb)[sk.kr], (uint64_t)d.wlo[kMaxCol + r], (uint32_t)tid,
                              FMT == kFmtTF32 ? TT_PREC_TF32 : FMT == kFmtFP16 ? TT_PREC_FP16 : TT_PREC_BF16);
          reinterpret_cast<float4*>(scale)[tid] = c;
        }
      }
    if (copies) {
      if (!*abort_flag) tc::mbar_wait(bar_g, gphase, abort_flag, status);   // bounded
      gphase ^= 1;
    }
    __syncthreads();
    if (t + 1 < ntile) {      // the next tile travels while this one is multiplied
      issue_x(a, td[nxt], raw, mi);
      cp_commit();
    }
    // the tile after that, in the slot of the one before this
    if (warp == kDescWarp && t + 2 < ntile) {
      if (lane == 0) advance();
      __syncwarp();
      describe(td[nxt == 2 ? 0 : nxt + 1], &td[nxt]);
    }
    // ---- column products of this warp's m-tile
    if (16 * warp < tak) {
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
            const uint32_t gs = s_u32(sm + a.col[s].soff) + (a.col[s].per ? mp * a.TB * LDG : 0);
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
    for (int q = 0; q < us.ntask[warp]; ++q) {
      const uint32_t gs = us.task[warp][q].gs;
      const int at = us.task[warp][q].acc, mtq = us.task[warp][q].mt;
      const int mt = mtq & 255;
      if (a.PR > 1 ? ((mtq >> 8) & 255) >= d.nr : 16 * mt >= d.tb) continue;
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
      float4* p = racc + d.gi * (a.nrow * mtB * NT * 32) + at + lane;
      const bool mbm = mtq >> 16;
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
    if (d.gi == ng - 1 && ++row_adds == kRowAddsMax) {
      row_adds = 0;
      __syncthreads();
      flush_rows();
    }
    if (t + 1 < ntile) cur = nxt;
  }
#pragma unroll
  for (int s = 0; s < NCOL; ++s)
    if (s < a.ncol) flush_col(s, td[cur].wlo[s]);
  __syncthreads();
  if (row_adds) flush_rows();
}

template <int FMT, int NT, int NCOL>
__global__ void __launch_bounds__(kThreads, NCOL * NT <= 12 ? 2 : 1)
    sketch_strip_kernel(const __grid_constant__ StripArgs a) {
  extern __shared__ __align__(16) char sm[];
  __shared__ TileDesc td[3];
  __shared__ UnitState us;
  __shared__ __align__(8) uint64_t bar;
  __shared__ int abort_flag;
  if (threadIdx.x == 0) {
    tc::mbar_init(s_u32(&bar), 1);
    abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  strip_unit<FMT, NT, NCOL, true>(a, blockIdx.x, sm, td, us, &bar, &abort_flag);
}

// Batched form: one launch over the units of every tensor of a plan, largest
// tensors first (prefix[] = first unit of each); the arguments of each tensor lie
// in the workspace, the split and the tensor pointers come by value (a captured launch
// needs nothing uploaded).
struct StripBatch {
  char* wsb;
  int64_t off_args;   // byte offset from wsb
  int nitems;
  uint32_t prefix[kMaxBatchItems + 1];
  const void* X[kMaxBatchItems];
};
template <int FMT, int NT>
__global__ void __launch_bounds__(kThreads, 2) sketch_strip_batched_kernel(const __grid_constant__ StripBatch b) {
  extern __shared__ __align__(16) char sm[];
  __shared__ TileDesc td[3];
  __shared__ UnitState us;
  __shared__ __align__(8) uint64_t bar;
  __shared__ int abort_flag;
  __shared__ __align__(16) StripArgs a;
  int lo = 0, hi = b.nitems - 1;   // position of the tensor of this unit (last prefix <= unit)
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (b.prefix[mid] <= blockIdx.x) lo = mid;
    else hi = mid - 1;
  }
  const uint32_t* src = reinterpret_cast<const uint32_t*>(b.wsb + b.off_args + (int64_t)lo * sizeof(StripArgs));
  for (int i = threadIdx.x; i < (int)(sizeof(StripArgs) / 4); i += kThreads) reinterpret_cast<uint32_t*>(&a)[i] = src[i];
  if (threadIdx.x == 0) {
    tc::mbar_init(s_u32(&bar), 1);
    abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    a.wsb = b.wsb;
    a.X = reinterpret_cast<const float*>(b.X[a.item]);
    a.vec = a.vec && ((uintptr_t)a.X & 15) == 0;
    const uint32_t ranges = (b.prefix[lo + 1] - b.prefix[lo]) / (uint32_t)(a.nA * a.nGS);
    a.CL = (a.npos + ranges - 1) / ranges;
  }
  __syncthreads();
  strip_unit<FMT, NT, kMaxCol, false>(a, blockIdx.x - b.prefix[lo], sm, td, us, &bar, &abort_flag);
}

using KernelFn = void (*)(const StripArgs);
using BatchFn = void (*)(const StripBatch);
// The instances of one format: column octets NT (smallest compiled one that
// holds nt) and NCOL = 2 or 3 column-sketch slots.
KernelFn kernel_bf16(int nt, int ncol);
KernelFn kernel_tf32(int nt, int ncol);
KernelFn kernel_fp16(int nt, int ncol);
BatchFn batched_bf16(int nt);   // nt = 2, 3 or 4
BatchFn batched_tf32(int nt);
BatchFn batched_fp16(int nt);
template <int FMT>
BatchFn batched_of(int nt) {
  return nt <= 2 ? sketch_strip_batched_kernel<FMT, 2> : nt == 3 ? sketch_strip_batched_kernel<FMT, 3>
                                                                 : sketch_strip_batched_kernel<FMT, 4>;
}
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
