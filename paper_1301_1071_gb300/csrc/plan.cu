// plan.cpp -- see plan.h.
#include "plan.h"

#include <algorithm>
#include <cstdint>
#include <numeric>

#include "../../include/tsqr.h"
#include "launch.h"
#include "layout.cuh"
#include "panel64.cuh"
#include "tc_kernels.cuh"

namespace tsqr {

static size_t al16(size_t x) { return (x + 15) / 16 * 16; }

// Workspace offsets with overflow checks: *ok is cleared when a sum or
// product does not fit in size_t (only sizes far beyond any device reach it).
static size_t add_ck(size_t a, size_t b, bool* ok) {
  if (a > SIZE_MAX - b) { *ok = false; return 0; }
  return a + b;
}
static size_t mul_ck(size_t a, size_t b, bool* ok) {
  if (b != 0 && a > SIZE_MAX / b) { *ok = false; return 0; }
  return a * b;
}
static size_t al16_ck(size_t x, bool* ok) {
  if (x > SIZE_MAX - 15) { *ok = false; return 0; }
  return al16(x);
}

// Register-tile heights and their thread bounds (must match tiles_f64.h and
// tiles_f32.h).  Each SM sub-partition holds 16K registers
// and a CTA of MAXT threads puts ceil(MAXT/128) warps on each, so the
// per-thread limit is 255 / 168 / 128 / 96 registers at MAXT = 256 / 384 /
// 512 / 640; R x 5 values (x2 registers for 8-byte and double-float values)
// leave about 60 registers for the rest of the kernel, with no spills.
// Tile 4 exceeds that budget (its registers spill); it is taken only when no
// other tile holds the rows asked for (binary64 tree nodes of two R factors
// at n > 64).  Tile 5 is wide: 8 columns per thread, 256 threads (n <= 64),
// taken exactly for 50 < n <= 64, where it beat the 5-column tiles (fewer
// warps sharing each column's reduction and reflector hand-off: 4,000,000 x
// 64 FP64 164.9 -> 114.1 ms, FP32 20.4 -> 18.1 ms); at n <= 50 its padded
// columns and fewer warps make it slower.
struct TileChoice { int R, maxt; bool spills; int npc; };
constexpr int kNumTiles = 7;
static const TileChoice kTiles64[kNumTiles] = {{16, 256, false, kNpc}, {10, 384, false, kNpc}, {6, 512, false, kNpc},
                                               {4, 640, false, kNpc},  {8, 640, true, kNpc},   {12, 256, false, 8},
                                               {5, 384, false, 10}};
static const TileChoice kTiles32[kNumTiles] = {{32, 256, false, kNpc}, {20, 384, false, kNpc}, {12, 512, false, kNpc},
                                               {8, 640, false, kNpc},  {16, 640, true, kNpc},  {24, 256, false, 8},
                                               {10, 384, false, 10}};
// columns per thread preferred for n
static int pref_npc(int n) { return n <= 50 ? kNpc : (n <= 64 ? 8 : 10); }

// Registers a thread may use under __launch_bounds__(maxt, 1): each of the
// 4 sub-partitions holds 16K registers for ceil(maxt / 128) warps.
static int reg_cap(int maxt) {
  const int w = (maxt + 127) / 128;
  int r = 16384 / (32 * w) / 8 * 8;
  return r > 255 ? 255 : r;
}

// Picks the register tile and row-group count.  want_b > 0: the smallest
// capacity B >= want_b (ties: the taller register tile); want_b == 0: the
// default policy below.
bool choose_cfg(int kind, int n, KernelCfg* out, int64_t want_b, int policy, int min_b) {
  if (n < 1 || n > TSQR_NMAX) return false;
  const int esz = kind == kKindF32 ? 4 : 8;
  const TileChoice* tiles = kind == kKindF32 ? kTiles32 : kTiles64;
  KernelCfg best;
  best.kind = kind;
  // pass 0: the tiles of this n's width; pass 1: any spill-free tile;
  // pass 2: the spilling tile.  A wanted capacity (want_b) considers both
  // widths from the start: the tightest fit wins.
  for (int pass = want_b > 0 ? 1 : 0; pass < 3 && best.B == 0; ++pass)
  for (int ti = 0; ti < kNumTiles; ++ti) {
    if (tiles[ti].spills != (pass == 2)) continue;
    if (pass == 0 && tiles[ti].npc != pref_npc(n)) continue;
    const int npc = tiles[ti].npc;
    const int CS = (n + npc - 1) / npc;
    const int NPAD = CS * npc;
    const int R = tiles[ti].R;
    for (int NRG = tiles[ti].maxt / (32 * CS); NRG >= 1; --NRG) {
      const int B = 32 * NRG * R;
      const int NT = 32 * CS * NRG;
      if (B < n || B < min_b) break;
      size_t a = LocalQrSmem(B, n, NT / 32, NPAD, esz, esz).total;
      if (a > kSmemMax) continue;
      int fq_rows = B;  // k_form_q stages its block in chunks of fq_rows rows
      while (fq_rows > 32 && FormQSmem(fq_rows, n, NPAD, esz, esz).total > kSmemMax) fq_rows -= 32;
      size_t f = FormQSmem(fq_rows, n, NPAD, esz, esz).total;
      if (f > kSmemMax) continue;
      int rm_rows = B;  // k_rowmul also stages two n x NPAD matrices: shrink its stage
      while (rm_rows > 32 && RowMulSmem(rm_rows, n, NPAD, esz, esz).total > kSmemMax) rm_rows -= 32;
      if (RowMulSmem(rm_rows, n, NPAD, esz, esz).total > kSmemMax) continue;
      // CTAs of k_local_qr per SM (register cap of the tile, shared memory)
      int ctas = 65536 / (NT * reg_cap(tiles[ti].maxt));
      const int by_smem = (int)(kSmemPerSM / (a + 1024));
      ctas = ctas < by_smem ? ctas : by_smem;
      ctas = ctas < 1 ? 1 : (ctas > 4 ? 4 : ctas);
      bool take;
      if (want_b > 0) {
        take = B >= want_b && (best.B == 0 || B < best.B || (B == best.B && R > best.R));
      } else if (policy == kPolicyLargest) {
        take = B > best.B;  // largest row block wins; ties keep the earlier tile
      } else if (policy == kPolicyInFlight) {
        const int64_t rows = (int64_t)B * ctas, best_rows = (int64_t)best.B * best.ctas;
        take = best.B == 0 || rows > best_rows || (rows == best_rows && ctas > best.ctas);
      } else {
        // Step 1: the largest block (the fixed per-column cost of the
        // Householder loop, and the per-tile cost of blocks of several tiles,
        // are spread over more rows; measured better than two smaller CTAs
        // per SM); ties: fewer threads
        take = best.B == 0 || B > best.B || (B == best.B && NT < best.NT);
      }
      if (take) {
        best.npc = npc; best.R = R; best.CS = CS; best.NRG = NRG; best.NT = NT; best.B = B;
        best.smem_qr = a; best.smem_fq = f; best.tile = ti; best.fq_rows = fq_rows;
        best.rm_rows = rm_rows; best.smem_rm = RowMulSmem(rm_rows, n, NPAD, esz, esz).total;
        best.ctas = ctas;
        // lanes reading one column of consecutive rows (row stride n elements)
        // fall into gcd(n words, 32) banks' worth of conflicts; 8-way or worse
        // is worth the rotated order (which spreads the n x NPAD coefficient
        // reads instead)
        best.skew = std::gcd(n * esz / 4, 32) >= 8 ? 1 : 0;
      }
    }
  }
  if (best.B == 0) return false;
  *out = best;
  return true;
}

// 16 warps of 128 registers an SM: as many CTAs as those and the shared memory
// allow (one ring slot is enough to run: it is held from publication to the
// last reader only), then ring slots up to one and a half a published panel.
PanelCfg choose_panel(int n) {
  PanelCfg c;
  c.NW = (n + kPdCols - 1) / kPdCols;
  // panel p takes p block reflectors and its own columns: weight p + 1, the
  // heaviest first to the sub-partition (warp w runs on w mod 4) with the least
  // work that has a warp left
  int load[4] = {0, 0, 0, 0}, used[4] = {0, 0, 0, 0};
  for (int p = c.NW - 1; p >= 0; --p) {
    int s = -1;
    for (int i = 0; i < 4; ++i)
      if (4 * used[i] + i < c.NW && (s < 0 || load[i] < load[s])) s = i;
    c.order |= static_cast<uint64_t>(p) << (4 * (4 * used[s] + s));
    load[s] += p + 1;
    ++used[s];
  }
  const int entries = c.NW - 1;  // published panels per tile
  for (c.ctas = kPdMaxThreads / 32 / c.NW; c.ctas >= 1; --c.ctas) {
    const size_t lim = c.ctas == 1 ? kSmemMax : kSmemPerSM / c.ctas - 1024;
    for (c.NS = entries + entries / 2 + 1; c.NS >= 1; --c.NS) {
      c.smem = Panel64Smem(c.NW, c.NS).total;
      if (c.smem <= lim) return c;
    }
  }
  return c;  // not reached: one CTA holds at least one slot for every n
}

GramGeom gram_geom(int64_t m, int n, int esz, bool small) {
  GramGeom g;
  int64_t chunk = (int64_t)(kSmemMax - 64) / (2 * (int64_t)n * esz);
  chunk = chunk > 1024 ? 1024 : chunk;
  chunk = chunk / 16 * 16;
  if (chunk < 16) chunk = 16;
  const bool digits = esz == 8 && n >= kSplitMinN && !small;
  if (digits) chunk = n <= 64 ? 64 : 32;  // k_gram_split
  g.chunk = (int)chunk;
  const int64_t nchunks = (m + chunk - 1) / chunk;
  const int most = digits ? kMaxGramParts64 : kMaxGramParts;
  g.grid = (int)(nchunks < most ? nchunks : most);
  const int n4 = (n + 3) / 4, n5 = (n + 4) / 5;
  g.tile = (n5 * n5 * 25 < n4 * n4 * 16) ? 5 : 4;  // fewer padded products
  const int nt1 = g.tile == 5 ? n5 : n4;
  int nt = (nt1 * nt1 + 31) / 32 * 32;
  g.nt = nt < 256 ? 256 : (nt > 1024 ? 1024 : nt);
  return g;
}

bool op_r_only(int op) { return op == TSQR_OP_R || op == TSQR_OP_SVD_VALUES || op == TSQR_OP_INDIRECT; }

size_t op_bytes(const Plan& P, int op) {
  return (op == TSQR_OP_CHOLQR || op == TSQR_OP_BACKWARD) ? P.bytes_gram : P.bytes;
}

int resolve_prec(int prec, int esz, int64_t n) {
  if (prec != TSQR_PREC_AUTO) return prec;
  // binary32 data: the Step-3 product on the tensor cores from n = 20 up,
  // where it outruns the FMA form; binary64 data: its one arithmetic, named
  // OZAKI for n <= 32
  if (esz == 4) return n >= kAutoTf32MinN ? TSQR_PREC_TF32X3 : TSQR_PREC_NATIVE;
  return n <= kOzMaxN ? TSQR_PREC_OZAKI : TSQR_PREC_NATIVE;
}

// Default block height of the panel form: k tiles a block for the least
// waves(k) k + 3.2 levels(k).  A tile costs a resident CTA about 3 n us through
// Steps 1 and 3 (n = 8 .. 64: 32, 63, 156, 200 us at n = 8, 25, 50, 64), a tree
// level about 9.5 n us (n = 25, 50, 64: 230, 465, 760).  30,000 x 50: one tile a
// block, 4 levels 2.27 ms, two tiles, 3 levels 1.88; 100,000 x 25: 3 levels
// 1.19 ms, 2 levels 0.89.  At most kMaxTiles tiles (the rounding of a block's
// chain grows with them).
static int64_t panel_block_rows(int64_t m, int64_t f, int64_t sms, int64_t slots, int64_t al) {
  auto levels = [&](int64_t p) {  // in rounds of a node an SM
    int64_t l = 0;
    for (; p > 1;) {
      p = (p + f - 1) / f;
      l += (p + sms - 1) / sms;
    }
    return l;
  };
  double best = 0;
  int64_t rows = kPdRows;
  for (int64_t k = 1; k <= kMaxTiles; ++k) {
    const int64_t p = (m + k * kPdRows - 1) / (k * kPdRows);
    const int64_t waves = (p + slots - 1) / slots;
    const double cost = (double)waves * (double)k + 3.2 * (double)levels(p);
    if (k == 1 || cost <= best) {  // taller blocks on a tie: fewer nodes (4,000,000 x 64 55.4 -> 53.2 ms)
      best = cost;
      rows = k * kPdRows;
      // blocks of even height over whole waves, where that adds no level
      const int64_t q = waves * slots;
      if (waves > 1 && levels(q) == levels(p)) {
        const int64_t b = (m + q - 1) / q;
        rows = (b + al - 1) / al * al;
      }
    }
    if (p == 1) break;
  }
  return rows;
}

static int plan_form(int64_t m, int64_t n, int esz, int64_t block_rows, int fanout, Plan* plan, int prec, int sms,
                     bool small, bool t_slots) {
  if (n < 1 || n > TSQR_NMAX || m < n) return TSQR_ERR_SHAPE;
  // every m x n matrix of the call, at 8 bytes an entry, must have a byte
  // size that int64 holds (the planner and the kernels index with it)
  if (m > INT64_MAX / 8 / n) return TSQR_ERR_SHAPE;
  prec = resolve_prec(prec, esz, n);
  if (prec != TSQR_PREC_NATIVE && !(prec == TSQR_PREC_DF64 && esz == 8) && !(prec == TSQR_PREC_TF32X3 && esz == 4) &&
      !(prec == TSQR_PREC_OZAKI && esz == 8))
    return TSQR_ERR_ARG;
  Plan P;
  P.m = m;
  P.n = n;
  P.esz = esz;
  const int kind0 = esz == 4 ? kKindF32 : (prec == TSQR_PREC_DF64 ? kKindDF64 : kKindF64);
  // Step-1 tile: the most rows resident per SM (double-float: the largest
  // tile); a smaller one when the caller's blocks fit in it
  const int policy0 = kind0 == kKindDF64 ? kPolicyStep1 : kPolicyInFlight;
  if (!choose_cfg(kind0, (int)n, &P.cfg0, 0, policy0) ||
      !choose_cfg(kKindF64, (int)n, &P.cfg64, 0, kPolicyStep1, 2 * (int)n))
    return TSQR_ERR_SHAPE;
  if (block_rows > 0 && block_rows <= P.cfg0.B && !choose_cfg(kind0, (int)n, &P.cfg0, block_rows, kPolicyStep1))
    return TSQR_ERR_SHAPE;
  // binary64 Step 1: panels of 8 columns, or the column-by-column register
  // tile (5 columns a warp) where that pads clearly less.  Step 1 of 3,000,000
  // rows, tile -> panels: n = 8 0.81 -> 0.72 ms, 10 0.87 -> 1.54, 12 1.75 -> 1.67,
  // 16 3.03 -> 1.88, 17 2.87 -> 3.40, 20 3.19 -> 3.74, 24 5.43 -> 3.85, 28 7.26 ->
  // 5.88, 32 10.96 -> 5.70, 48 30.9 -> 11.5 (2,000,000 rows 7.64, and 6.33 since the
  // panels are dealt evenly).  At the line, whole calls of 3,000,000 rows, direct
  // and R alone, tile / panels: n = 20 4.79 and 3.05 / 6.11 and 3.70, 25 7.61 and
  // 5.11 / 8.38 and 5.31, 33 15.3 and 10.2 / 14.0 and 7.2, 35 15.8 and 10.5 / 14.6
  // and 7.6: beyond 25 the tile holds fewer rows and panels win whatever they pad
  P.panel = kind0 == kKindF64 && n >= kSplitMinN && !small &&
            !(n <= 25 && (n + 4) / 5 * 5 + 3 < (n + kPdCols - 1) / kPdCols * kPdCols);
  if (P.panel) P.pq = choose_panel((int)n);
  if (sms > 0) P.pq.sms = sms;
  P.B0 = P.panel ? kPdRows : P.cfg0.B;
  P.ctas0 = P.panel ? P.pq.ctas : P.cfg0.ctas;
  const int64_t B0 = P.B0;
  // rows per tile after the first: the register tile less the carried R,
  // rounded down so that every tile starts on a 16-byte boundary when the
  // block does (bulk copies)
  int64_t al = 1;
  while ((al * n * esz) % 16 != 0) ++al;
  // (the panel form keeps R out of the tile)
  const int64_t bt = (P.panel ? B0 : B0 - n) / al * al;
  if (bt < 1) return TSQR_ERR_SHAPE;
  // tree node = f stacked R factors, f >= 2: up to the binary64 row-block
  // tile's rows (fmax), or any f whose node fits one CTA's shared memory or
  // a cluster of f CTAs.  Default: fmax, at most kTreeMaxF (a node's chain grows
  // with its triangles: 100,000 x 10 in 100 blocks 372 us at f = 100, 314 at 10;
  // 124,103 x 8 391 us at f = 256, 229 at 32), while that is kTreeClMaxF or
  // more; else nodes of kTreeClMaxF triangles on clusters (1,000,000 x 64: 12.4 ms
  // at f = 6, 10.8 at 8; 20,000,000 x 100 has 4 tree levels instead of 10); then
  // (where 4 triangles fit one CTA) the least fan-in that needs no more levels
  // (608 blocks of n = 64: 4 levels at f = 8 and at 5, 9.13 against 8.47 ms)
  const int64_t fmax = P.cfg64.B / n;
  const int ni = static_cast<int>(n);
  int64_t f = fanout;
  if (fanout <= 0)
    f = small ? (fmax >= 4 && tree_up_fits(ni, 4) ? fmax : kTreeClMaxF)
              : (fmax >= kTreeClMaxF && tree_up_fits(ni, 4) ? std::min(fmax, kTreeMaxF) : kTreeClMaxF);
  int64_t b0 = block_rows;
  if (b0 <= 0 && P.panel) {
    b0 = panel_block_rows(m, f, P.pq.sms, (int64_t)P.pq.sms * P.ctas0, al);
  } else if (b0 <= 0) {
    if (sms < 1) sms = kDefaultSMs;
    const int64_t kmax = kind0 == kKindDF64 ? kMaxTilesDF64 : (kind0 == kKindF32 ? kMaxTilesF32 : kMaxTiles);
    const int64_t bmax = B0 + (kmax - 1) * bt;
    if (m <= (int64_t)kMinWaves * sms * P.ctas0 * B0) {
      b0 = B0;
    } else {
      const int64_t slots = (int64_t)sms * P.ctas0;  // CTAs resident at once
      int64_t waves = (m + slots * bmax - 1) / (slots * bmax);
      const int64_t wmin = (kMinWaves + P.ctas0 - 1) / P.ctas0;  // kMinWaves blocks per SM
      if (waves < wmin) waves = wmin;
      const int64_t p = waves * slots;
      b0 = (m + p - 1) / p;
      b0 = (b0 + al - 1) / al * al;  // blocks start on 16-byte boundaries
    }
  }
  if (b0 < n) return TSQR_ERR_SHAPE;
  if (b0 > m) b0 = m;  // one block
  if (fanout <= 0 && !small && tree_up_fits(ni, 4)) {
    auto levels = [&](int64_t g) {
      int l = 0;
      for (int64_t p = (m + b0 - 1) / b0; p > 1; p = (p + g - 1) / g) ++l;
      return l;
    };
    // (narrow triangles: one level takes up to kTreeOneLevelF of them -- 40 or 79
    // blocks at n = 3 .. 16 in one level 0.80 to 0.91 of the time in two)
    const int64_t p = (m + b0 - 1) / b0;
    if (n <= kTreeNarrowN && p <= std::min(fmax, kTreeOneLevelF) && tree_up_fits(ni, static_cast<int>(p)))
      f = std::max<int64_t>(f, p);
    const int l = levels(f);
    while (f > 2 && levels(f - 1) == l) --f;
  }
  const int64_t kt0 = b0 <= B0 ? 1 : 1 + (b0 - B0 + bt - 1) / bt;
  // tiles per block: more of the panel form's short ones, for the heights of the other
  if (kt0 > (P.panel ? 1 << 24 : 1 << 20)) return TSQR_ERR_SHAPE;
  if (f < 2 || (f > fmax && !tree_up_fits(ni, static_cast<int>(f)) && !tree_up_cl_fits(ni, static_cast<int>(f))))
    return TSQR_ERR_SHAPE;

  P.prec = prec;
  P.tc3 = prec == TSQR_PREC_TF32X3 && n <= kTcwMaxN;
  P.oz3 = prec == TSQR_PREC_OZAKI && n >= kSplitMinN && n <= kOzMaxN;
  // binary64 arithmetic: Step 3 and (Step 1's one-row-group tiles) the T
  // factors' Gram as exact digit products
  P.split3 = kind0 == kKindF64 && rows_by_digits(n);
  P.gram_split = kind0 == kKindF64 && n >= kSplitMinN && (P.panel || P.cfg0.NRG == 1);
  P.fuse_sign = P.gram_split && !P.oz3;
  P.rows32 = esz == 4 && step3_rows32((int)n, (m + b0 - 1) / b0, P.pq.sms);
  {
    const int kind_rm = esz == 4 ? kKindF32 : kKindF64;
    // the coefficient blocks' padded width: the wider of the two tile widths'
    // paddings (the tile chosen below may be either)
    const int NPAD = (int)std::max(std::max((n + kNpc - 1) / kNpc * kNpc, (n + 7) / 8 * 8), (n + 9) / 10 * 10);
    int64_t b2 = 32;
    while (RowMulSmem((int)(2 * (b2 + 32)), (int)n, NPAD, esz, esz).total <= kSmemMax) b2 += 32;
    if (RowMulSmem((int)(2 * b2), (int)n, NPAD, esz, esz).total > kSmemMax) return TSQR_ERR_SHAPE;
    // the smallest tile holding b2 rows, else (small n) the largest tile
    if (!choose_cfg(kind_rm, (int)n, &P.cfg_rm2, b2, kPolicyStep1) &&
        !choose_cfg(kind_rm, (int)n, &P.cfg_rm2, 0, kPolicyLargest))
      return TSQR_ERR_SHAPE;
    P.b_rm2 = P.cfg_rm2.B < b2 ? P.cfg_rm2.B : b2;
    P.cfg_rm2.rm_rows = (int)(2 * P.b_rm2);
    P.cfg_rm2.smem_rm = RowMulSmem(P.cfg_rm2.rm_rows, (int)n, P.cfg_rm2.CS * P.cfg_rm2.npc, esz, esz).total;
  }
  Level l0;
  l0.rows = m;
  l0.b = b0;
  l0.p = (m + b0 - 1) / b0;
  l0.bt = bt;
  l0.kt = (int)kt0;
  P.levels.push_back(l0);
  while (P.levels.back().p > 1) {
    Level l;
    l.rows = P.levels.back().p * n;
    l.b = f * n;
    l.p = (l.rows + l.b - 1) / l.b;
    l.bt = P.cfg64.B - n;  // tree nodes fit one tile (f n <= B)
    l.kt = 1;
    P.levels.push_back(l);
  }
  // The kernels take a block's height as int and launch one CTA per row
  // block, per T slot (the T build) or per triangle of a tree node (cluster
  // nodes): heights and grids beyond int and gridDim.x (2^31 - 1) are shape
  // errors here rather than truncated launch arguments.
  if (b0 > INT32_MAX) return TSQR_ERR_SHAPE;
  for (size_t i = 0; i < P.levels.size(); ++i) {
    const Level& l = P.levels[i];
    if (l.p > INT32_MAX / l.kt || (i > 0 && l.p > INT32_MAX / f)) return TSQR_ERR_SHAPE;
  }
  bool ok = true;
  size_t o = kHeaderBytes;
  const size_t nn = (size_t)n * n * sizeof(double);
  for (auto& l : P.levels) {
    l.off_S = o;
    o = al16_ck(add_ck(o, mul_ck((size_t)l.p, nn, &ok), &ok), &ok);
    l.off_T = o;
    if (t_slots) o = al16_ck(add_ck(o, mul_ck(mul_ck((size_t)l.p, (size_t)l.kt, &ok), nn, &ok), &ok), &ok);
  }
  P.off_ctop = o;
  o = al16_ck(add_ck(o, nn, &ok), &ok);
  P.off_small = o;
  o = al16_ck(add_ck(o, kSmallSlots * nn, &ok), &ok);
  P.bytes = o;
  GramGeom g = gram_geom(m, (int)n, esz, small);
  P.gram_chunk = g.chunk;
  P.gram_grid = g.grid;
  P.gram_nt = g.nt;
  o = kHeaderBytes;
  P.off_part = o;
  o = al16(o + (size_t)g.grid * nn);
  P.off_gsmall = o;
  o = al16(o + kSmallSlots * nn);
  P.bytes_gram = o;
  if (!ok) return TSQR_ERR_SHAPE;
  *plan = P;
  return TSQR_OK;
}

// Whether the tiles of the small plan S take less time than the panels of F, by
// the chain that one CTA and the tree run through, in n us.  Few blocks (at most
// one an SM): a tile of 320 or 512 rows in one CTA against two to five panel
// tiles, which the panel plan joins to save a tree level.  A panel tile takes
// 4.4 the first (n = 16 .. 64: 62, 99, 141, 194, 308 us at 16, 22, 32, 40, 64), 3.2
// each further one, with Step 3 by FMAs (n > 64) 10; a column tile of R rows a
// thread 0.28 R + 0.2 + 0.065 n (n = 11, 32, 50, 64: 40, 219, 300, 530); a level 5 to
// 8.5 (up, T, down).  10,000 x 11: panels 232 us, tiles 163; 40,000 x 50 2.11 ms and
// 1.63; 3,000 x 92 4.93 and 3.70; 130 x 65 1.10 and 0.76; 10,000 x 64 panels 1.82, tiles
// 2.12.
static bool tiles_faster(const Plan& F, const Plan& S, int64_t sms) {
  const Level &a = F.levels[0], &b = S.levels[0];
  if (a.kt < 2 || b.kt != 1 || b.p > sms) return false;
  const double n = (double)F.n, level = 5.0 + 0.14 * std::min(n, 25.0);
  const double panel = (4.4 + (F.n <= kRowSplitMaxN ? 3.2 : 10.0) * (a.kt - 1)) * (kPdCols * F.pq.NW / n);
  const double tile = 1.12 * (0.28 * S.cfg0.R + 0.2 + 0.065 * n);
  return tile + level * (double)(S.levels.size() - 1) < panel + level * (double)(F.levels.size() - 1);
}

int make_plan(int64_t m, int64_t n, int esz, int64_t block_rows, int fanout, Plan* plan, int prec, int sms, bool small,
              bool t_slots) {
  int rc = TSQR_ERR_SHAPE;
  if (!small) rc = plan_form(m, n, esz, block_rows, fanout, plan, prec, sms, false, t_slots);
  // the sizes that the taller tiles take or refuse (block heights of 2^20 tiles,
  // 2^31 T slots) are those of either form, so that they do not move with it
  constexpr int64_t kFarM = int64_t(1) << 24;
  Plan alt;
  if (rc == TSQR_ERR_SHAPE) return plan_form(m, n, esz, block_rows, fanout, plan, prec, sms, true, t_slots);
  if (rc == TSQR_OK && plan->panel && m >= kFarM)
    rc = plan_form(m, n, esz, block_rows, fanout, &alt, prec, sms, true, t_slots);
  else if (rc == TSQR_OK && plan->panel && block_rows <= 0 && plan->levels[0].kt > 1 &&
           plan_form(m, n, esz, block_rows, fanout, &alt, prec, sms, true, t_slots) == TSQR_OK &&
           tiles_faster(*plan, alt, plan->pq.sms))
    *plan = alt;
  return rc;
}

int make_host_plan(int64_t m, int64_t n, int esz, int64_t block_rows, int fanout, Plan* plan, int* chunks,
                   int prec, int sms, bool small) {
  Plan P0;
  int rc = make_plan(m, n, esz, block_rows, fanout, &P0, prec, sms, small);
  if (rc != TSQR_OK) return rc;
  if (sms < 1) sms = kDefaultSMs;
  const int64_t slots = (int64_t)sms * P0.ctas0;
  if (block_rows <= 0) {
    int64_t c = (m * n * esz) / kHostChunkBytes;
    c = c < 1 ? 1 : (c > kMaxHostChunks ? kMaxHostChunks : c);
    if (c > 1) {
      // c chunks of w waves each, blocks no taller than the default plan's
      const int64_t p0 = P0.levels[0].p;
      const int64_t w = (p0 + c * slots - 1) / (c * slots);
      const int64_t p = c * slots * (w < 1 ? 1 : w);
      int64_t al = 1;
      while ((al * n * esz) % 16 != 0) ++al;
      int64_t b = (m + p - 1) / p;
      b = (b + al - 1) / al * al;
      if (b >= n && b >= P0.B0) {
        Plan P1;
        if (make_plan(m, n, esz, b, fanout, &P1, prec, sms, small) == TSQR_OK) P0 = P1;
      }
    }
  }
  const int64_t p = P0.levels[0].p;
  int64_t c = p / slots;
  c = c < 1 ? 1 : (c > kMaxHostChunks ? kMaxHostChunks : c);
  *chunks = (int)c;
  *plan = P0;
  return TSQR_OK;
}

}  // namespace tsqr
