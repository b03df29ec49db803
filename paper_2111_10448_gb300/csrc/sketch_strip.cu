// Strip kernel (strip.cuh): host side.
//
// The fused multi-sketch for shapes outside the tcgen05
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
// What bounds it: issue slots, of which 54 % are used (96^4 x 6; 16 warps an SM leave
// barriers and dependent chains uncovered).  At 96^4 x 48, l = 28, leaving one part out
// saved: the normals 7.6 of 32.7 ms (5.3 since they take fewer slots), the rest of the
// staging 5, conversion 4, copies of X 2, column products 2.2, row products 3.7.
// mma.sync itself (1015 FMA per cycle and SM measured in 16 bits, 2 d round8(l) FMAs an
// entry) is busy 15 %.
//
// Measured (one accumulate, BF16 unless named; the 64 x 32 tile kernel that served
// these shapes before in brackets): 960^3, l = 35: 3.32 ms (13.0); 64^5, l = 28:
// 7.5 ms (26); 300^3, l = 60: 0.362 ms (0.79), TF32 0.51 (0.87); 200 x 128 x 100 x
// 80, l = 16, FP16 Khatri-Rao: 1.03 ms (4.33); 16 x 300 x 300: 0.048 ms (0.150).
// 24^6, l = 26: 2.70 ms (small-plane kernel: 10.7); 96^4 x 48, l = 28: 30.0.
// No shape tried was slower, down to 8^3, 9 x 9 x 1000 and 2 x 1000 x 1000, so every
// call with one to three sketches a side takes it (d <= 6 two-sided, d <= 4
// one-sided; more accumulators than that do not fit the registers and the
// small-plane and 64 x 32 kernels stay, as for plans with no sketch on one side:
// one-sided two-pass and d = 2 two-pass; and for Khatri-Rao small planes).
//
// Precision: 32 of the contraction are a chain of 4 MMA instructions (8 in TF32), the
// low part of each k-step first; chains are summed in FP32 round-to-nearest, at most kAddsMax
// = 12 on the column side and 64 on the row side (16 visits of up to 4), then in FP64.
#include <algorithm>
#include <cstring>

#include "strip.cuh"

namespace tts {

const DevSketch* plan_sketches_host(const Plan* p);

namespace strip {
namespace {

constexpr int kSmemTwo = 111 * 1024;   // dynamic shared memory of a CTA, two per SM
constexpr int kSmemOne = 224 * 1024;   // one per SM
// Quads of normals that pay for staging them: 2.6 us at 2.0e11 a second, a launch.  Sketch
// with every shared row staged -> with this: 16^4 47 -> 40 us, 9^6 TF32 172 -> 161, 4 x 30 x 30 x
// 30 x 5 106 -> 92, 512 x 512 45 -> 39; 24^6 and 960^3 stage as before.
constexpr int64_t kTableQuads = 1 << 19;
// Entries of a batched unit: the whole batch over about four units per CTA slot, at least
// kUnitMin (the row sums of a unit are an FP64 atomic each) and at most kUnitMax.  A batch
// whose tensors were cut into units of 2^17 whatever their number left most of the slots
// without one.  Calls of 2 tensors of 10^5 entries, 8 of 10^6, 64 of 10^5, 512 of 10^6 (BF16): 511, 639,
// 623, 10540 us so, now 154, 318, 402, 10628; the small-plane kernel, tuned, 187, 579, 659, 32300.
constexpr int64_t kUnitMin = 1 << 11, kUnitMax = 1 << 17, kUnitStep = 1 << 11;

int strip_octets(const Plan& P, int item) {
  const DevItem& it = plan_items_host(&P)[item];
  const DevSketch* sks = plan_sketches_host(&P);
  int lmax = 1;
  for (int s = 0; s < it.nsk; ++s) lmax = std::max(lmax, sks[it.sk0 + s].width);
  return strip_nt(lmax);
}

// Fills the launch arguments when the kernel serves this call.
// nt_batch: column octets of a batched launch (0: a launch of its own), whose units are
// sized when it is launched (*units: the least number of them).
bool plan_strip(const Plan& P, int item, int64_t count, StripArgs* out, int* fmt_out, int* nt_out, size_t* smem,
                int64_t* units, int nt_batch = 0) {
  const DevItem& it = plan_items_host(&P)[item];
  if (it.x_f64 || (it.prec != TT_PREC_BF16 && it.prec != TT_PREC_TF32 && it.prec != TT_PREC_FP16)) return false;
  const int fmt = it.prec == TT_PREC_TF32 ? kFmtTF32 : it.prec == TT_PREC_FP16 ? kFmtFP16 : kFmtBF16;
  const DevSketch* sks = plan_sketches_host(&P);
  StripArgs g;
  memset(&g, 0, sizeof(g));
  bool kr = false;
  for (int s = 0; s < it.nsk; ++s) {
    const DevSketch& d = sks[it.sk0 + s];
    StSk k;
    memset(&k, 0, sizeof(k));
    k.rows = d.rows;
    k.off = d.off;
    k.hstride = d.hstride;
    k.tab = d.st_tab;
    if (d.wdiv >= (1LL << 31)) return false;
    if (!nt_batch && k.tab >= 0) {
      // quads drawn without the table (a row per tile row that reads it) less those it holds
      const bool col = d.type == SK_COL;
      const int64_t rows = col ? it.W / d.wdiv * count : d.wdiv * it.n[0];
      const int64_t uses = col ? d.wdiv * ((it.n[0] + kMaxTA - 1) / kMaxTA) : it.W / d.wdiv * ((count + 63) / 64);
      if ((uses - 1) * rows * ((d.width + 3) / 4) < kTableQuads) k.tab = -1;
    }
    k.wdiv = (uint32_t)d.wdiv;
    k.width = d.width;
    k.nq = (d.width + 3) / 4;
    k.inv_nq = 1.0f / (float)k.nq;
    k.rpi = kThreads / k.nq;
    k.sid = d.stream_id;
    k.kr = d.kr_nm ? it.sk0 + s : -1;
    k.mbm = d.kr_nm && d.kr_mbm ? 1 : 0;
    kr = kr || d.kr_nm;
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
  const int nt = nt_batch ? nt_batch : strip_octets(P, item);
  const int64_t nrh = it.d - 1 > it.ds ? it.n[it.d - 2] : 1, sR = WR / nrh, q2 = it.ds >= 2 ? it.n[1] : 1;
  for (int s = 0; s < g.ncol; ++s) g.tabs |= g.col[s].tab >= 0 ? 1u << s : 0u;
  for (int r = 0; r < g.nrow; ++r) g.tabs |= g.row[r].tab >= 0 ? 1u << (kMaxCol + r) : 0u;
  for (int s = 0; s < g.ncol; ++s) {
    const int64_t w = g.col[s].wdiv;
    if (w != 1 && w != q2 && w != WL) return false;
    g.col[s].kind = w == WL ? 2 : w == 1 ? 0 : 1;
    g.col[s].mulr = WL / w;
  }
  for (int r = 0; r < g.nrow; ++r) {
    const int64_t q = g.row[r].wdiv / WL;
    if (q != 1 && q != sR && q != WR) return false;
    g.row[r].kind = q == WR ? 2 : q == 1 ? 0 : 1;
  }
  g.n1 = it.n[0];
  g.cnt = count;
  g.Nd1 = it.N[it.d - 1];
  g.seed = it.seed;
  g.keys = philox_keys(it.seed);
  g.xscale = fmt == kFmtFP16 ? it.xscale : 1.0f;
  g.WL = (uint32_t)WL;
  g.WR = (uint32_t)WR;
  g.q2 = (uint32_t)q2;
  g.q3 = it.ds >= 3 ? (uint32_t)it.n[2] : 1u;
  g.nrh = (uint32_t)nrh;
  g.sR = (uint32_t)sR;
  // strips and tiles of even size, rounded to m-tiles
  g.nA = (int)((g.n1 + kMaxTA - 1) / kMaxTA);
  g.n1p = (int)(((g.n1 + g.nA - 1) / g.nA + 15) / 16 * 16);
  g.nA = (int)((g.n1 + g.n1p - 1) / g.n1p);
  g.nB = (int)((count + tbmax - 1) / tbmax);
  g.ndp = (int)(((count + g.nB - 1) / g.nB + 15) / 16 * 16);
  g.nB = (int)((count + g.ndp - 1) / g.ndp);
  const int E = esz(fmt), ldg = ldg_bytes(fmt, nt);
  const int ncs = nt_batch || g.ncol > 2 ? 3 : 2;
  // shared memory before the row sums, and one column tile's row sums
  auto layout = [&](int PL, int PR, int* per) {
    g.PL = PL;
    g.PR = PR;
    g.TA = PL * g.n1p;
    g.TB = PR * g.ndp;
    int off = g.TB * (g.TA + 8) * E;
    g.off_xl = off;
    off *= 2;
    g.off_raw = off;
    const int run = PL > 1 ? PL * (int)g.n1 : g.n1p;
    g.rawld = (run + 3) / 4 * 4 + 4;
    off += PR * (int)std::min<int64_t>(count, g.ndp) * g.rawld * 4;
    g.off_g = off;
    for (int s = 0; s < g.ncol; ++s) {
      g.col[s].per = PL > 1 && g.col[s].wdiv == 1 ? 1 : 0;
      g.col[s].soff = off;
      off += (g.col[s].per ? PL : 1) * g.TB * ldg;
    }
    for (int r = 0; r < g.nrow; ++r) {
      g.row[r].per = PR > 1 && g.row[r].wdiv == (uint32_t)it.W ? 1 : 0;
      g.row[r].soff = off;
      off += (g.row[r].per ? PR : 1) * g.TA * ldg;
    }
    g.off_scale = off;
    off += 8 * nt * (int)sizeof(float);
    g.off_acc = (off + 15) / 16 * 16;
    *per = g.nrow * (g.TB / 16) * nt * 512;
    return g.off_acc;
  };
  // Small planes are grouped into tiles (dense test matrices only: a mode-by-mode
  // sketch is scaled per plane): the largest tile that leaves two CTAs an SM.
  const bool regs_two = ncs * nt <= 12;
  int PL = 1, PR = 1, per = 0;
  if (!kr && (g.nA == 1 || g.nB == 1)) {
    int64_t best = 0;
    const int pl_max = g.nA == 1 ? (int)std::min<int64_t>(kMaxTA / g.n1p, g.q2) : 1;
    const int pr_max = g.nB == 1 ? (int)std::min<int64_t>(std::max<int64_t>(1, tbmax / g.ndp), g.nrh) : 1;
    for (int pl = 1; pl <= pl_max; ++pl)
      for (int pr = 1; pr <= pr_max; ++pr) {
        if (layout(pl, pr, &per) + per > (regs_two ? kSmemTwo : kSmemOne)) continue;
        const int64_t area = (int64_t)pl * pr;
        if (area > best || (area == best && pl * g.n1p >= pr * g.ndp && PL * g.n1p < PR * g.ndp)) {
          best = area;
          PL = pl;
          PR = pr;
        }
      }
  }
  int off = layout(PL, PR, &per);
  g.inv_pl = 1.0f / (float)PL;
  g.npos = (uint32_t)((g.q2 + PL - 1) / PL * g.q3);
  g.ngt = (uint32_t)(g.sR * ((g.nrh + PR - 1) / PR) * g.nB);
  // the row sums of a set of column tiles take the rest; fewer when the sets
  // alone would leave SMs without a unit
  const int mtA = g.TA / 16, mtB = g.TB / 16;
  const int slots = device_sm_count() * 2;
  const bool two = regs_two && off + per <= kSmemTwo;
  int64_t ng = ((two ? kSmemTwo : kSmemOne) - off) / per;
  if (ng < 1) return false;
  ng = std::min<int64_t>(ng, g.ngt);
  if (!nt_batch) ng = std::min(ng, std::max<int64_t>(1, (int64_t)g.ngt * g.nA * g.npos / slots));
  g.nGS = (int)((g.ngt + ng - 1) / ng);
  g.NG = (int)((g.ngt + g.nGS - 1) / g.nGS);
  g.nGS = (int)((g.ngt + g.NG - 1) / g.NG);
  // position ranges: about four units per CTA slot
  const int64_t base = (int64_t)g.nA * g.nGS;
  const int64_t goal = nt_batch ? base : 4LL * slots;
  const int64_t want = std::max<int64_t>(1, std::min<int64_t>(g.npos, (goal + base - 1) / base));
  g.CL = (uint32_t)((g.npos + want - 1) / want);
  *units = base * ((g.npos + g.CL - 1) / g.CL);
  if (*units >= (1LL << 31)) return false;
  // row products (m-tile, sketch) to the least-loaded warp; a warp with an
  // m-tile of the strip starts with its column products
  int load[kWarps], cnt[kWarps];
  for (int w = 0; w < kWarps; ++w) {
    load[w] = (w < mtA ? g.ncol * g.TB : 0) + (w == kDescWarp ? kDescLoad : 0);
    cnt[w] = 0;
    memset(g.task[w], 255, kWarpTasks);
  }
  for (int mt = 0; mt < mtB; ++mt)
    for (int r = 0; r < g.nrow; ++r) {
      int w = 0;
      for (int v = 1; v < kWarps; ++v)
        if (cnt[v] < kWarpTasks && (cnt[w] == kWarpTasks || load[v] < load[w])) w = v;
      g.task[w][cnt[w]++] = (uint8_t)(mt + 8 * r);
      load[w] += g.TA;
    }
  g.item = item;
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
  g.cpr = g.rawld / 4;
  g.total = g.Nd1 * count;
  int ic = 0, ir = 0;
  for (int s = 0; s < it.nsk; ++s) {
    const DevSketch& d = sks[it.sk0 + s];
    if ((d.type == SK_COL ? g.col[ic++] : g.row[ir++]).tab < 0) continue;
    // stage the sketch's rows for this call, in the kernel's own row format: the
    // slab's i_d (column side) or i_1 (row side)
    const bool col = d.type == SK_COL;
    const int lpad = strip::ldg_bytes(fmt, nt) / strip::esz(fmt);
    const cudaError_t e = launch_rows_table(d, it.sk0 + s, (const char*)ws, it.seed, first, it.n[0],
                                            col ? (int)count : (int)it.n[0], lpad, col ? it.W / d.wdiv : d.wdiv,
                                            (char*)ws + d.st_tab, it.prec, true, st);
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

namespace {
// Units of one tensor of a batch, of about `unit` entries each: base x equal ranges of its
// positions (sketch_strip_batched_kernel takes the ranges' length from this count).
int64_t units_of(const StripBatchItem& it, int64_t unit) {
  const int64_t goal = (it.entries + unit - 1) / unit;
  const int64_t want = std::max<int64_t>(1, std::min<int64_t>(it.npos, (goal + it.base - 1) / it.base));
  const int64_t len = (it.npos + want - 1) / want;
  return it.base * ((it.npos + len - 1) / len);
}
}  // namespace

bool strip_plan_batched(const Plan& P, const std::vector<int>& order, StripBatchPlan* out) {
  int64_t units = 0;
  const int n = plan_num_items(&P);
  out->args.clear();
  out->items.clear();
  out->entries = 0;
  out->nt = 2;
  out->smem = 0;
  if (n < 2 || n > kMaxBatchItems) return false;
  for (int i = 0; i < n; ++i) {
    const DevItem& it = plan_items_host(&P)[i];
    if (it.prec != plan_items_host(&P)[0].prec || it.sptab_doubles == 0) return false;
    out->nt = std::max(out->nt, strip::strip_octets(P, i));
  }
  if (out->nt > 4) return false;
  out->args.resize((size_t)n * sizeof(strip::StripArgs));
  for (int pos = 0; pos < n; ++pos) {
    strip::StripArgs g;
    int fmt, nt;
    size_t smem;
    int64_t u;
    const DevItem& it = plan_items_host(&P)[order[(size_t)pos]];
    if (!strip::plan_strip(P, order[(size_t)pos], it.n[it.d - 1], &g, &fmt, &nt, &smem, &u, out->nt)) return false;
    if (smem > (size_t)strip::kSmemTwo) return false;
    g.vec = it.n[0] % 4 == 0;
    g.cpr = g.rawld / 4;
    g.total = g.Nd1 * g.cnt;
    std::memcpy(out->args.data() + (size_t)pos * sizeof(g), &g, sizeof(g));
    out->smem = std::max(out->smem, smem);
    out->items.push_back(StripBatchItem{it.N[it.d], (uint32_t)u, g.npos});
    out->entries += it.N[it.d];
    // the finest split of every tensor has to fit a launch
    if (units_of(out->items.back(), strip::kUnitMin) + units >= (1LL << 31)) return false;
    units += units_of(out->items.back(), strip::kUnitMin);
  }
  return true;
}

cudaError_t launch_sketch_strip_batched(const Plan& P, const StripBatchPlan& bp, int64_t off_args, const BatchCfg& cfg,
                                        const void* const* X, void* ws, cudaStream_t st) {
  const int n = plan_num_items(&P);
  const int prec = plan_items_host(&P)[0].prec;
  const int fmt = prec == TT_PREC_TF32 ? strip::kFmtTF32 : prec == TT_PREC_FP16 ? strip::kFmtFP16 : strip::kFmtBF16;
  cudaError_t e = cudaMemsetAsync((char*)ws + kStatusOff, 0, sizeof(int), st);
  if (e != cudaSuccess) return e;
  const int lpad = strip::ldg_bytes(fmt, bp.nt) / strip::esz(fmt);
  e = launch_rows_table_batched((char*)ws, n, lpad, st);
  if (e != cudaSuccess) return e;
  strip::StripBatch b;
  b.wsb = (char*)ws;
  b.off_args = off_args;
  b.nitems = n;
  // a shape set by hand or by the tuner, else from the batch
  const int64_t unit = cfg.ta <= 8 ? strip::kUnitStep * std::min<int64_t>(64, (int64_t)cfg.ta * cfg.chunk)
                                   : std::min<int64_t>(strip::kUnitMax, std::max<int64_t>(
                                         strip::kUnitMin, bp.entries / (8LL * device_sm_count())));
  b.prefix[0] = 0;
  for (int i = 0; i < n; ++i) b.prefix[i + 1] = b.prefix[i] + (uint32_t)units_of(bp.items[(size_t)i], unit);
  std::memcpy(b.X, X, sizeof(void*) * (size_t)n);
  const strip::BatchFn k = fmt == strip::kFmtTF32   ? strip::batched_tf32(bp.nt)
                           : fmt == strip::kFmtFP16 ? strip::batched_fp16(bp.nt)
                                                    : strip::batched_bf16(bp.nt);
  static bool attr_set[3][5] = {};
  if (!attr_set[fmt][bp.nt]) {
    e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, strip::kSmemTwo);
    if (e != cudaSuccess) return e;
    attr_set[fmt][bp.nt] = true;
  }
  count_launch();
  k<<<b.prefix[n], strip::kThreads, bp.smem, st>>>(b);
  return cudaGetLastError();
}

}  // namespace tts
