// Strip kernel (strip.cuh): host side.
//
// The fused multi-sketch for shapes outside the tcgen05 and small-plane
// kernels: X = stack of planes X(:, w, :), w = kL + WL kR, every entry of X
// read once and fed to every sketch (internal.cuh states the products).
//
// Split of the work.  Column-sketch rows depend on (i_1, kL), row-sketch rows on
// (kR, i_d).  A CTA takes one strip of i_1 (at most 128 rows), a set of column
// tiles (kR, block of i_d) and a range of kL values, and walks the set for each
// kL.  The column sums of the strip stay in registers (one 16-row m-tile per
// warp) while the set is walked, and go to the FP64 sketch when kL moves
// their rows on; the row sums of the whole set stay in shared memory over all
// kL of the unit.  So an FP64 atomic is paid per (set width) entries on the
// column side and per (kL range) x (strip) entries on the row side, instead of
// once per 64 x 32 tile.  A tile of X is converted to hi and lo parts once, in one
// shared-memory layout that both products read through ldmatrix; a test-matrix
// block is staged again only when its rows change (Omega_{d*} per column tile,
// Psi_{d*} per kL, ...).  The next tile is copied to shared memory
// (cp.async) while this one is multiplied; two CTAs per SM overlap one's staging
// with the other's products.
//
// What bounds it: mma.sync (1015 FMA per cycle and SM measured in 16 bits):
// 2 d round8(l) FMAs an entry.
//
// Measured (one accumulate, BF16 unless named; the 64 x 32 tile kernel that served
// these shapes before in brackets): 960^3, l = 35: 3.45 ms (13.0); 64^5, l = 28:
// 9.3 ms (26); 300^3, l = 60: 0.36 ms (0.79), TF32 0.55 (0.87); 200 x 128 x 100 x
// 80, l = 16, FP16 Khatri-Rao: 1.08 ms (4.33); 16 x 300 x 300: 0.071 ms (0.150).
// No shape tried was slower, down to 9 x 9 x 1000 and 2 x 1000 x 1000, so every
// call with at most three sketches a side takes it (d <= 6 two-sided, d <= 4
// one-sided; more accumulators than that do not fit the registers and the
// 64 x 32 kernel stays).
//
// Precision: MMA chains of at most 4 instructions (32 of the contraction, hi and
// lo), summed in FP32 round-to-nearest over at most kAddsMax of them, then FP64.
#include <algorithm>
#include <cstring>

#include "strip.cuh"

namespace tts {

const DevSketch* plan_sketches_host(const Plan* p);

namespace strip {
namespace {

constexpr int kSmemTwo = 111 * 1024;   // dynamic shared memory of a CTA, two per SM
constexpr int kSmemOne = 224 * 1024;   // one per SM

uint32_t recip20(int d) { return ((1u << 20) + (uint32_t)d - 1u) / (uint32_t)d; }

int nt_instance(int nt) { return nt <= 2 ? 2 : nt <= 6 ? nt : 8; }

// Fills the launch arguments when the kernel serves this call.
bool plan_strip(const Plan& P, int item, int64_t count, StripArgs* out, int* fmt_out, int* nt_out, size_t* smem,
                int64_t* units) {
  const DevItem& it = plan_items_host(&P)[item];
  if (it.x_f64 || (it.prec != TT_PREC_BF16 && it.prec != TT_PREC_TF32 && it.prec != TT_PREC_FP16)) return false;
  const int fmt = it.prec == TT_PREC_TF32 ? kFmtTF32 : it.prec == TT_PREC_FP16 ? kFmtFP16 : kFmtBF16;
  const DevSketch* sks = plan_sketches_host(&P);
  StripArgs g;
  memset(&g, 0, sizeof(g));
  int lmax = 1;
  for (int s = 0; s < it.nsk; ++s) {
    const DevSketch& d = sks[it.sk0 + s];
    StSk k;
    memset(&k, 0, sizeof(k));
    k.rows = d.rows;
    k.off = d.off;
    k.hstride = d.hstride;
    k.tab = d.gen_tab >= 0 && it.gentab_doubles > 0 ? it.off_gentab * 8 + d.gen_tab : -1;
    if (d.wdiv >= (1LL << 31)) return false;
    k.wdiv = (uint32_t)d.wdiv;
    k.width = d.width;
    k.lpad = (d.width + 15) / 16 * 16;
    k.sid = d.stream_id;
    k.kr = d.kr_nm ? it.sk0 + s : -1;
    k.mbm = d.kr_nm && d.kr_mbm ? 1 : 0;
    lmax = std::max(lmax, d.width);
    if (d.type == SK_COL) {
      if (g.ncol == kMaxCol) return false;
      g.col[g.ncol++] = k;
    } else {
      if (g.nrow == kMaxRow) return false;
      g.row[g.nrow++] = k;
    }
  }
  if (!g.ncol || !g.nrow || it.ds > 3) return false;
  const int64_t WL = it.N[it.ds] / it.n[0], WR = it.W / WL;
  const int64_t tbmax = fmt == kFmtTF32 ? 32 : 64;
  if (it.n[0] >= (1LL << 31) || count < 1 || count >= (1LL << 31) || it.W >= (1LL << 31) ||
      WR * ((count + tbmax - 1) / tbmax) >= (1LL << 31))
    return false;
  const int nt = nt_instance((lmax + 7) / 8);
  g.n1 = it.n[0];
  g.cnt = count;
  g.Nd1 = it.N[it.d - 1];
  g.seed = it.seed;
  g.xscale = fmt == kFmtFP16 ? it.xscale : 1.0f;
  g.WL = (uint32_t)WL;
  g.WR = (uint32_t)WR;
  g.q2 = it.ds >= 2 ? (uint32_t)it.n[1] : 1u;
  g.q3 = it.ds >= 3 ? (uint32_t)it.n[2] : 1u;
  // strips and tiles of even size, rounded to m-tiles
  g.nA = (int)((g.n1 + kMaxTA - 1) / kMaxTA);
  g.TA = (int)(((g.n1 + g.nA - 1) / g.nA + 15) / 16 * 16);
  g.nA = (int)((g.n1 + g.TA - 1) / g.TA);
  g.nB = (int)((count + tbmax - 1) / tbmax);
  g.TB = (int)(((count + g.nB - 1) / g.nB + 15) / 16 * 16);
  g.nB = (int)((count + g.TB - 1) / g.TB);
  g.ngt = (uint32_t)(WR * g.nB);
  const int E = esz(fmt), mtB = g.TB / 16, mtA = g.TA / 16;
  int off = g.TB * (g.TA + 8) * E;
  g.off_xl = off;
  off *= 2;
  g.off_raw = off;
  off += g.TB * (g.TA + 4) * 4;
  for (int s = 0; s < g.ncol; ++s) {
    g.col[s].soff = off;
    off += g.TB * ldg_bytes(fmt, nt);
  }
  for (int r = 0; r < g.nrow; ++r) {
    g.row[r].soff = off;
    off += g.TA * ldg_bytes(fmt, nt);
  }
  g.off_scale = off;
  off += 8 * nt * (int)sizeof(float);
  g.off_acc = off = (off + 15) / 16 * 16;
  // the row sums of a set of column tiles take the rest; fewer when the sets
  // alone would leave SMs without a unit
  const int per = g.nrow * mtB * nt * 512;
  const int slots = device_sm_count() * 2;
  const bool two = (g.ncol <= 2 ? 2 : 3) * nt <= 12 && off + per <= kSmemTwo;
  int64_t ng = ((two ? kSmemTwo : kSmemOne) - off) / per;
  if (ng < 1) return false;
  ng = std::min<int64_t>(ng, g.ngt);
  ng = std::min(ng, std::max<int64_t>(1, (int64_t)g.ngt * g.nA * WL / slots));
  g.nGS = (int)((g.ngt + ng - 1) / ng);
  g.NG = (int)((g.ngt + g.nGS - 1) / g.nGS);
  g.nGS = (int)((g.ngt + g.NG - 1) / g.NG);
  // kL ranges: about four units per CTA slot
  const int64_t base = (int64_t)g.nA * g.nGS;
  const int64_t want = std::max<int64_t>(1, std::min<int64_t>(WL, (4LL * slots + base - 1) / base));
  g.CL = (uint32_t)((WL + want - 1) / want);
  *units = base * ((WL + g.CL - 1) / g.CL);
  if (*units >= (1LL << 31)) return false;
  g.inv_qpr = recip20(g.TA / 4);
  // row products (m-tile, sketch) to the least-loaded warp; a warp with an
  // m-tile of the strip starts with its column products
  int load[kWarps], cnt[kWarps];
  for (int w = 0; w < kWarps; ++w) {
    load[w] = w < mtA ? g.ncol * g.TB : 0;
    cnt[w] = 0;
    memset(g.task[w], 255, kMaxTasks);
  }
  for (int mt = 0; mt < mtB; ++mt)
    for (int r = 0; r < g.nrow; ++r) {
      int w = 0;
      for (int v = 1; v < kWarps; ++v)
        if (load[v] < load[w]) w = v;
      g.task[w][cnt[w]++] = (uint8_t)(mt + 8 * r);
      load[w] += g.TA;
    }
  *out = g;
  *fmt_out = fmt;
  *nt_out = nt;
  *smem = (size_t)g.off_acc + (size_t)g.NG * per;
  return true;
}

}  // namespace
}  // namespace strip

bool use_strip_kernel(const Plan& P, int item, int64_t count) {
  strip::StripArgs g;
  int fmt, nt;
  size_t smem;
  int64_t units;
  return strip::plan_strip(P, item, count, &g, &fmt, &nt, &smem, &units);
}

cudaError_t launch_sketch_strip(const Plan& P, int item, const void* X, int64_t first, int64_t count, void* ws,
                                cudaStream_t st) {
  strip::StripArgs g;
  int fmt, nt;
  size_t smem;
  int64_t units;
  if (!strip::plan_strip(P, item, count, &g, &fmt, &nt, &smem, &units)) return cudaErrorNotSupported;
  const DevItem& it = plan_items_host(&P)[item];
  const DevSketch* sks = plan_sketches_host(&P);
  g.X = (const float*)X;
  g.wsb = (char*)ws;
  g.first = first;
  g.vec = it.n[0] % 4 == 0 && ((uintptr_t)X & 15) == 0 ? 1 : 0;
  g.cpr = g.TA / 4 + (g.vec ? 0 : 1);
  g.inv_cpr = strip::recip20(g.cpr);
  g.total = g.Nd1 * count;
  for (int s = 0; s < it.nsk; ++s) {
    const DevSketch& d = sks[it.sk0 + s];
    if (d.gen_tab < 0 || it.gentab_doubles == 0) continue;
    // stage the sketch's rows for this call: the slab's i_d (column side) or i_1 (row side)
    const bool col = d.type == SK_COL;
    const cudaError_t e = launch_rows_table(d, it.sk0 + s, (const char*)ws, it.seed, first, it.n[0],
                                            col ? (int)count : (int)it.n[0], (d.width + 15) / 16 * 16,
                                            col ? it.W / d.wdiv : d.wdiv, (char*)ws + it.off_gentab * 8 + d.gen_tab,
                                            it.prec, st);
    if (e != cudaSuccess) return e;
  }
  const strip::KernelFn k = fmt == strip::kFmtTF32   ? strip::kernel_tf32(nt, g.ncol)
                            : fmt == strip::kFmtFP16 ? strip::kernel_fp16(nt, g.ncol)
                                                     : strip::kernel_bf16(nt, g.ncol);
  static bool attr_set[3][9][2] = {};
  bool& set = attr_set[fmt][nt][g.ncol <= 2 ? 0 : 1];
  if (!set) {
    const cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, strip::kSmemOne);
    if (e != cudaSuccess) return e;
    set = true;
  }
  count_launch();
  k<<<(unsigned)units, strip::kThreads, smem, st>>>(g);
  return cudaGetLastError();
}

}  // namespace tts
