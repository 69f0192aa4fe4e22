// split_kernels.cuh -- the tall binary64 products as exact digit products on
// the tensor cores (split.cuh): rows times an n x n matrix, and Grams.
#pragma once

#include <cstdint>
#include <type_traits>

#include "device.cuh"
#include "layout.cuh"
#include "split.cuh"

namespace tsqr {

// Shared memory of k_rowmul_split: M's digit fragments, exponents, and per
// warp a buffer of 16 rows with its mbarrier.  One buffer is enough: the rows
// are in registers as digits before the products start, and the next tile's
// copy runs behind those.
constexpr int kRsThreads = 256;
constexpr int kRsRows = 16;
constexpr int kRsMaxN = 64;
struct RowSplitSmem {
  size_t b, cexp, kexp, bars, rows, total, buf;
  TSQR_HD RowSplitSmem(int n) {
    size_t o = 0;
    b = o; o = align_up(o + split_b_bytes(n), 128);
    cexp = o; o = align_up(o + 8 * split_nt(n) * sizeof(int), 16);
    kexp = o; o = align_up(o + 16 * split_kc(n) * sizeof(int), 16);
    bars = o; o = align_up(o + (kRsThreads / 32) * 8, 128);
    buf = align_up(static_cast<size_t>(kRsRows) * n * 8, 128);
    rows = o; o += (kRsThreads / 32) * buf;
    total = o;
  }
};

// out_r (+)= X_r M for every row r (M n x n, n <= 64).  colsrc != NULL: an
// n x n upper-triangular matrix R with X = Q R for a well-scaled Q: column k
// of X is taken relative to the largest entry of column k of R (its own
// scale), so that badly scaled columns keep their digits; colexp != NULL: the
// columns' largest exponents themselves (split_exp).  add: to what `out` holds.
// X may be out (each 16-row tile is read before it is written).
//
// Bound by the integer unit: per entry about 14 operations to split it and, per
// output, about 32 to recombine it.  A warp per 16 rows (the fragment's height),
// rows by bulk copy one tile ahead.  8,000,000 x 25: 8.02 ms by binary64 FMAs,
// 2.19 so (its 3.2 GB 0.48); 4,000,000 x 64, two products: 56.1 and 9.0.
template <int KC>
__global__ void __launch_bounds__(kRsThreads, KC <= 2 ? 2 : 1)
    k_rowmul_split(const double* X, const double* __restrict__ M, const double* __restrict__ colsrc,
                   const int* __restrict__ colexp, int64_t m, int n, bool add, double* out, int32_t* status) {
  extern __shared__ __align__(128) unsigned char smem[];
  const RowSplitSmem L(n);
  uint2* bfrag = reinterpret_cast<uint2*>(smem + L.b);
  int* cexp = reinterpret_cast<int*>(smem + L.cexp);
  int* kx = reinterpret_cast<int*>(smem + L.kexp);
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + L.bars);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int g = lane >> 2, t = lane & 3;
  if (threadIdx.x == 0) {
    for (int i = 0; i < kRsThreads / 32; ++i) mbar_init(bars + i, 1);
    fence_mbar_init();
  }
  const bool scaled = colsrc != nullptr || colexp != nullptr;
  for (int k = threadIdx.x; k < 16 * KC; k += kRsThreads) {
    int e = kExpZero;
    if (k < n) {
      if (colsrc)
        for (int i = 0; i <= k; ++i) e = max(e, split_exp(colsrc[static_cast<int64_t>(i) * n + k]));
      else if (colexp)
        e = colexp[k];
    }
    kx[k] = e == kExpZero ? 0 : e;
  }
  __syncthreads();
  split_build_b([&](int k, int c) { return M[static_cast<int64_t>(k) * n + c]; }, n, KC, scaled ? kx : nullptr, cexp,
                bfrag);
  __syncthreads();
  const int NT = split_nt(n);
  const int64_t nt = (m + kRsRows - 1) / kRsRows;
  const int64_t stride = static_cast<int64_t>(gridDim.x) * (kRsThreads / 32);
  int64_t tile = static_cast<int64_t>(blockIdx.x) * (kRsThreads / 32) + warp;
  double* xs = reinterpret_cast<double*>(smem + L.rows + static_cast<size_t>(warp) * L.buf);
  uint64_t* bar = bars + warp;
  // rows of a tile: one bulk copy (its start is a multiple of 128 n bytes; the
  // last tile's odd 8 bytes by a plain load)
  auto issue = [&](int64_t ti) {
    if (ti < nt && lane == 0) {
      const int64_t r0 = ti * kRsRows;
      const int rows = static_cast<int>(m - r0 < kRsRows ? m - r0 : kRsRows);
      const uint32_t bytes = static_cast<uint32_t>(rows) * n * 8, body = bytes & ~15u;
      if (body != bytes) xs[body / 8] = X[r0 * n + body / 8];
      mbar_arrive_expect_tx(bar, body);
      if (body) bulk_g2s(xs, X + r0 * n, body, bar);
    }
  };
  issue(tile);
  uint32_t ph = 0;
  for (; tile < nt; tile += stride) {
    if (!mbar_wait_bounded(bar, ph)) {
      if (lane == 0) set_status(status, TSQR_ERR_TIMEOUT);
      return;
    }
    ph ^= 1u;
    __syncwarp();
    const int64_t r0 = tile * kRsRows;
    const int rows = static_cast<int>(m - r0 < kRsRows ? m - r0 : kRsRows);
    uint32_t a[KC][8][4];
    int er[2];
    bool bad[2];
    split_rows<KC>([&](int r, int k) { return (r < rows && k < n) ? xs[r * n + k] : 0.0; }, n, scaled ? kx : nullptr,
                   a, er, bad);
    __syncwarp();  // every lane has its rows: the buffer takes the next tile
    issue(tile + stride);
    for (int j = 0; j < NT; ++j) {
      long long o[4];
      int oe[4];
      split_product<KC>(a, bfrag + static_cast<size_t>(j) * KC * 8 * 32, lane, o, oe);
      const int c0 = 8 * j + 2 * t;
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int r = g + 8 * h;
        if (r < rows && c0 < n) {
          double* q = out + (r0 + r) * n + c0;
          double v[2];
#pragma unroll
          for (int i = 0; i < 2; ++i) {
            const int ce = cexp[c0 + i];
            v[i] = split_to_double(o[2 * h + i], er[h] + ce + oe[2 * h + i] - kSplitShift);
            if (bad[h] || ce == kExpBad) v[i] = __longlong_as_double(0x7ff8000000000000ll);
          }
          if (c0 + 1 < n && (n & 1) == 0) {
            double2* q2 = reinterpret_cast<double2*>(q);
            double2 w = make_double2(v[0], v[1]);
            if (add) {
              const double2 p = *q2;
              w.x += p.x;
              w.y += p.y;
            }
            *q2 = w;
          } else {
            q[0] = add ? q[0] + v[0] : v[0];
            if (c0 + 1 < n) q[1] = add ? q[1] + v[1] : v[1];
          }
        }
      }
    }
  }
}

// ---------------------------------------------------------------------------
// Step 3 (Sec. III-B) for binary64 data with n <= 64: Q_i = Q1_i C_i, tiles
// last to first with X = C as in k_form_q -- tile t >= 1: W = T X, rows -V_t W,
// X <- X - W; tile 0: W = T (Y_top^T X), rows [X; 0] - Y W -- with T X and V W
// as digit products.  One CTA per row block; a warp per 16 rows.
// Bound by the integer unit (splitting, recombining) and, for n > 32, the
// tensor products; T X through the binary64 unit would cost more than all rows
// of a tile (n = 64: 74,000 cycles against 43,000).  1,000,003 x 25: 1.34 ms by
// binary64 FMAs, 0.48 so (0.4 GB: 0.06); 4,000,000 x 64: 38.9 and 8.7 (4.1 GB: 0.61).
// ---------------------------------------------------------------------------
struct FormQSplitSmem {
  size_t b, x, w, cexp, bars, rows, total, buf;
  TSQR_HD FormQSplitSmem(int n) {
    size_t o = 0;
    b = o; o = align_up(o + split_b_bytes(n), 128);
    x = o; o = align_up(o + static_cast<size_t>(n) * n * 8, 16);
    w = o; o = align_up(o + static_cast<size_t>(n) * n * 8, 16);
    cexp = o; o = align_up(o + 8 * split_nt(n) * sizeof(int), 16);
    bars = o; o = align_up(o + (kRsThreads / 32) * 8, 128);
    buf = align_up(static_cast<size_t>(kRsRows) * n * 8, 128);
    rows = o; o += (kRsThreads / 32) * buf;
    total = o;
  }
};

template <int KC>
__global__ void __launch_bounds__(kRsThreads, KC <= 2 ? 2 : 1)
    k_form_q_split(double* Yg, int64_t m, int n, int b, int B, int bt, int kt, const double* __restrict__ Tg,
                   const double* __restrict__ Cg, int64_t cblocks, bool comp, int32_t* status) {
  extern __shared__ __align__(128) unsigned char smem[];
  const FormQSplitSmem L(n);
  uint2* bfrag = reinterpret_cast<uint2*>(smem + L.b);
  double* xm = reinterpret_cast<double*>(smem + L.x);
  double* wm = reinterpret_cast<double*>(smem + L.w);
  int* cexp = reinterpret_cast<int*>(smem + L.cexp);
  constexpr int NWARP = kRsThreads / 32;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int g = lane >> 2, t2 = 2 * (lane & 3);
  double* ys = reinterpret_cast<double*>(smem + L.rows + static_cast<size_t>(warp) * L.buf);
  uint64_t* bar = reinterpret_cast<uint64_t*>(smem + L.bars) + warp;
  if (threadIdx.x < NWARP) mbar_init(reinterpret_cast<uint64_t*>(smem + L.bars) + threadIdx.x, 1);
  fence_mbar_init();
  const int64_t row0 = static_cast<int64_t>(blockIdx.x) * b;
  const int rows = static_cast<int>(m - row0 < b ? m - row0 : b);
  const int ntiles = row_tiles(rows, B, bt);
  const int ntop = rows < n ? rows : n;
  const int nn = n * n, NT = split_nt(n);
  const double* Cb = Cg + (cblocks == 1 ? 0 : static_cast<int64_t>(blockIdx.x)) * nn;
  for (int e = threadIdx.x; e < nn; e += kRsThreads) xm[e] = Cb[e];
  __syncthreads();

  // this warp's row pieces: pieces warp, warp + 8, .. of each tile, tiles last
  // to first; (pt, pr) is the next one to copy
  auto tile_rows = [&](int t, int& tr0, int& cnt) {
    tr0 = t == 0 ? 0 : B + (t - 1) * bt;
    cnt = t == 0 ? (rows < B ? rows : B) : (rows - tr0 < bt ? rows - tr0 : bt);
  };
  int pt = ntiles - 1, pr = warp * kRsRows;
  auto issue = [&]() {
    int tr0 = 0, cnt = 0;
    for (; pt >= 0; --pt, pr = warp * kRsRows) {
      tile_rows(pt, tr0, cnt);
      if (pr < cnt) break;
    }
    if (pt < 0) return;
    const int rc = cnt - pr < kRsRows ? cnt - pr : kRsRows;
    const double* src = Yg + (row0 + tr0 + pr) * n;
    const uint32_t bytes = static_cast<uint32_t>(rc) * n * 8;
    const uint32_t body = (reinterpret_cast<uintptr_t>(src) & 15) == 0 ? bytes & ~15u : 0u;
    for (uint32_t e = body / 8 + lane; e < bytes / 8; e += 32) ys[e] = src[e];  // a ragged or unaligned piece
    if (lane == 0) {
      mbar_arrive_expect_tx(bar, body);
      if (body) bulk_g2s(ys, src, body, bar);
    }
    pr += kRsRows * NWARP;
  };
  issue();
  uint32_t ph = 0;
  bool ok = true;
  for (int t = ntiles - 1; t >= 0; --t) {
    int tr0, cnt;
    tile_rows(t, tr0, cnt);
    const bool top = t == 0;
    const double* Tb = Tg + (static_cast<int64_t>(blockIdx.x) * kt + t) * nn;
    const double* src = xm;
    if (top) {
      // Z = Y_top^T X (Y_top unit lower triangular; no row is overwritten yet)
      for (int e = threadIdx.x; e < nn; e += kRsThreads) {
        const int kk = e / n, c = e - kk * n;
        double s = 0.0;
        if (kk < ntop) {
          s = xm[e];
          for (int r = kk + 1; r < ntop; ++r) s = fma(Yg[(row0 + r) * n + kk], xm[r * n + c], s);
        }
        wm[e] = s;
      }
      __syncthreads();
      src = wm;
    }
    split_build_b([&](int k, int c) { return src[k * n + c]; }, n, KC, nullptr, cexp, bfrag);
    __syncthreads();
    // W = T src, tau_i src_i in binary64 and the strict triangle as digit
    // products: T is close to 2 I in a block's later tiles, so the triangle's
    // own scale is far below tau's and X keeps its relative accuracy through
    // hundreds of X <- X - W (all of T in one scale doubled Q's error).  Warp w
    // takes T's rows 16 (w mod KC) .., columns by the rest
    {
      constexpr int SHARE = NWARP / KC;
      const int rt = warp % KC, part = warp / KC;
      if (part < SHARE) {
        uint32_t a[KC][8][4];
        int er[2];
        bool bad[2];
        split_rows<KC>(
            [&](int r, int k) {
              const int i = 16 * rt + r;
              return (i < n && k < n && k > i) ? Tb[static_cast<int64_t>(i) * n + k] : 0.0;
            },
            n, nullptr, a, er, bad);
        for (int j = part; j < NT; j += SHARE) {
          long long o[4];
          int oe[4];
          split_product<KC>(a, bfrag + static_cast<size_t>(j) * KC * 8 * 32, lane, o, oe);
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const int r = 16 * rt + g + 8 * (i >> 1), c = 8 * j + t2 + (i & 1);
            if (r < n && c < n) {
              double v = split_to_double(o[i], er[i >> 1] + cexp[c] + oe[i] - kSplitShift);
              if (bad[i >> 1] || cexp[c] == kExpBad) v = __longlong_as_double(0x7ff8000000000000ll);
              const double tau = Tb[static_cast<int64_t>(r) * n + r], xo = src[r * n + c];
              wm[r * n + c] = fma(tau, xo, v);
              // the coefficient of tile t - 1, X - W = -X + ((2 - tau) X - v):
              // with tau close to 2 one rounding of X a tile
              if (!top) xm[r * n + c] = fma(comp ? Tb[comp_at(r, n)] : 2.0 - tau, xo, -v) - xo;
            }
          }
        }
      }
    }
    __syncthreads();
    split_build_b([&](int k, int c) { return wm[k * n + c]; }, n, KC, nullptr, cexp, bfrag);
    __syncthreads();
    for (int p0 = warp * kRsRows; p0 < cnt; p0 += kRsRows * NWARP) {
      ok = ok && mbar_wait_bounded(bar, ph);
      ph ^= 1u;
      if (!ok) {
        if (lane == 0) set_status(status, TSQR_ERR_TIMEOUT);
        break;
      }
      __syncwarp();
      const int rc = cnt - p0 < kRsRows ? cnt - p0 : kRsRows;
      double* q = Yg + (row0 + tr0 + p0) * n;
      uint32_t a[KC][8][4];
      int er[2];
      bool bad[2];
      split_rows<KC>(
          [&](int r, int k) {
            if (top && k >= p0 + r && k < n) return k == p0 + r && p0 + r < ntop ? 1.0 : 0.0;
            return (r < rc && k < n) ? ys[r * n + k] : 0.0;
          },
          n, nullptr, a, er, bad);
      __syncwarp();
      issue();
      for (int j = 0; j < NT; ++j) {
        long long o[4];
        int oe[4];
        split_product<KC>(a, bfrag + static_cast<size_t>(j) * KC * 8 * 32, lane, o, oe);
        const int c0 = 8 * j + t2;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int r = g + 8 * h;
          if (r < rc && c0 < n) {
            double v[2];
#pragma unroll
            for (int i = 0; i < 2; ++i) {
              const int ce = cexp[c0 + i];
              v[i] = split_to_double(-o[2 * h + i], er[h] + ce + oe[2 * h + i] - kSplitShift);
              if (bad[h] || ce == kExpBad) v[i] = __longlong_as_double(0x7ff8000000000000ll);
              if (top && p0 + r < ntop && c0 + i < n) v[i] += xm[(p0 + r) * n + c0 + i];
            }
            double* d = q + r * n + c0;
            if ((n & 1) == 0) {
              *reinterpret_cast<double2*>(d) = make_double2(v[0], v[1]);
            } else {
              d[0] = v[0];
              if (c0 + 1 < n) d[1] = v[1];
            }
          }
        }
      }
    }
    __syncthreads();  // the fragments are rebuilt for the next tile
  }
}

// ---------------------------------------------------------------------------
// Grams X^T Y (X == Y: symmetric, the tiles on and above the diagonal only).
// One warp per 8-column group loads CR rows of it (a lane the column pair 2 t
// of rows g, g + 8, ..), takes the columns' largest exponents over the chunk,
// and writes the 8 balanced digits (62-bit fixed point) to planes of 16-byte
// rows, from which ldmatrix.trans gives both operands' fragments: the products
// contract over rows.  Each warp then forms its 16 x 8 output tiles -- 36 digit
// products a k step -- and folds a chunk's integers into binary64.
// X^T X of 8,000,000 x 25: 8.37 ms by binary64 FMAs, 1.65 so (1.6 GB: 0.24);
// X^T Y of 4,000,000 x 64: 26.8 and 4.9.  Bound by the integer unit's splitting and,
// from n = 49 on, by the products of one CTA an SM.
//
// TM = false: G = X^T Y over all rows, chunk by chunk round the CTAs; the
// CTA's n x n partial goes to part.  colexp != NULL: the columns' largest
// exponents of X (atomicMax, zeroed by the caller).
// TM = true: X holds the Householder vectors of Step 1; the Gram of every
// tile goes to the strictly upper triangle of its T slot (items: tiles).
// ---------------------------------------------------------------------------
struct GramSplitSmem {
  size_t px, py, ex, ey, total;
  int ncg, nca;  // 8-column groups, rounded up to even (the A operand takes two)
  TSQR_HD GramSplitSmem(int n, int CR, bool sym) {
    ncg = (n + 7) / 8;
    nca = (ncg + 1) & ~1;
    const size_t plane = static_cast<size_t>(8) * nca * CR * 16;
    size_t o = 0;
    px = o; o += plane;
    py = sym ? px : o; o += sym ? 0 : plane;
    ex = o; o += static_cast<size_t>(nca) * 8 * sizeof(int);
    ey = sym ? ex : o; o += sym ? 0 : static_cast<size_t>(nca) * 8 * sizeof(int);
    total = align_up(o, 16);
  }
};

template <class S, bool SYM, bool TM, int CR, int TW, int MAXT, int MINB>
__global__ void __launch_bounds__(MAXT, MINB)
    k_gram_split(const S* __restrict__ X, const S* __restrict__ Yin, int64_t m, int n, double* part,
                 int* colexp, int64_t b, int B, int bt, int kt, int64_t p) {
  static_assert(!TM || SYM, "the T factors' Gram is symmetric");
  extern __shared__ __align__(128) unsigned char smem[];
  constexpr int RL = CR / 8;  // row groups of 8 per chunk
  const GramSplitSmem L(n, CR, SYM);
  int* ex = reinterpret_cast<int*>(smem + L.ex);
  int* ey = reinterpret_cast<int*>(smem + L.ey);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, NW = blockDim.x >> 5;  // NW = ncg
  const int g = lane >> 2, t = lane & 3;
  const uint32_t pxa = smem_u32(smem + L.px), pya = smem_u32(smem + L.py);
  // the padding group's planes stay zero
  for (int i = threadIdx.x; i < (L.nca - L.ncg) * 8 * CR; i += blockDim.x) {
    const int d = i / CR, r = i - d * CR;
    const size_t off = (static_cast<size_t>(d * L.nca + L.ncg) * CR + r) * 16;
    *reinterpret_cast<uint4*>(smem + L.px + off) = make_uint4(0, 0, 0, 0);
    if (!SYM) *reinterpret_cast<uint4*>(smem + L.py + off) = make_uint4(0, 0, 0, 0);
  }
  for (int i = threadIdx.x; i < L.nca * 8; i += blockDim.x) ex[i] = ey[i] = 0;
  __syncthreads();

  const int c0 = 8 * warp + 2 * t;  // this lane's column pair in the loads
  const bool wide = (n & 1) == 0;   // pairs of entries are aligned
  using S2 = typename std::conditional<sizeof(S) == 8, double2, float2>::type;
  auto load = [&](const S* src, int64_t r0, int rows, double (&v)[RL][2], int top) {
#pragma unroll
    for (int i = 0; i < RL; ++i) {
      const int r = 8 * i + g;
      v[i][0] = v[i][1] = 0.0;
      if (r < rows && c0 < n) {
        const S* q = src + (r0 + r) * n + c0;
        if (wide) {
          const S2 w = *reinterpret_cast<const S2*>(q);
          v[i][0] = w.x;
          v[i][1] = w.y;
        } else {
          v[i][0] = q[0];
          if (c0 + 1 < n) v[i][1] = q[1];
        }
        if (TM && top + r < n) {  // tile 0's top rows: unit lower triangular
#pragma unroll
          for (int k = 0; k < 2; ++k)
            if (c0 + k >= top + r) v[i][k] = c0 + k == top + r ? 1.0 : 0.0;
        }
      }
    }
  };
  int runmax[2] = {kExpZero, kExpZero};
  auto split = [&](const double (&v)[RL][2], uint32_t plane, int* es, bool track) {
    int em[2] = {kExpZero, kExpZero};
#pragma unroll
    for (int i = 0; i < RL; ++i)
#pragma unroll
      for (int k = 0; k < 2; ++k) em[k] = max(em[k], split_exp(v[i][k]));
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      em[k] = max(em[k], __shfl_xor_sync(0xffffffffu, em[k], 4));
      em[k] = max(em[k], __shfl_xor_sync(0xffffffffu, em[k], 8));
      em[k] = max(em[k], __shfl_xor_sync(0xffffffffu, em[k], 16));
      if (track) runmax[k] = max(runmax[k], em[k]);
    }
    if (lane < 4) {
      es[c0] = em[0];
      es[c0 + 1] = em[1];
    }
#pragma unroll
    for (int i = 0; i < RL; ++i) {
      long long f[2];
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        const int e = static_cast<int>((static_cast<uint32_t>(__double2hiint(v[i][k])) >> 20) & 0x7ffu);
        f[k] = split_fixed<62>(v[i][k], max(em[k] - (e > 0 ? e : 1), 0));
      }
      uint32_t h[8];
      split_digits(f[0], f[1], h);
#pragma unroll
      for (int d = 0; d < 8; ++d)
        asm volatile("st.shared.b32 [%0], %1;" ::"r"(plane + ((d * L.nca + warp) * CR + 8 * i + g) * 16 + 4 * t),
                     "r"(h[d])
                     : "memory");
    }
  };

  // output tiles (16 columns mi of X, 8 columns nj of Y) of this warp
  const int nmi = L.nca / 2;
  int tmi[TW], tnj[TW];
  {
    int k = 0, idx = 0;
#pragma unroll
    for (int u = 0; u < TW; ++u) tmi[u] = -1, tnj[u] = 0;
    for (int mi = 0; mi < nmi; ++mi)
      for (int nj = SYM ? 2 * mi : 0; nj < L.ncg; ++nj, ++idx)
        if (idx % NW == warp) {
#pragma unroll
          for (int u = 0; u < TW; ++u)
            if (u == k) tmi[u] = mi, tnj[u] = nj;
          ++k;
        }
  }
  double sum[TW][4];
#pragma unroll
  for (int u = 0; u < TW; ++u)
#pragma unroll
    for (int i = 0; i < 4; ++i) sum[u][i] = 0.0;
  auto products = [&]() {
#pragma unroll
    for (int u = 0; u < TW; ++u) {
      if (tmi[u] < 0) continue;
      float acc[8][4], ac2[4][4];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
#pragma unroll
        for (int d = 0; d < 8; ++d) acc[d][i] = kSplitMagic;
#pragma unroll
        for (int d = 0; d < 4; ++d) ac2[d][i] = kSplitMagic;
      }
      const int mat = lane >> 3, mr = lane & 7;
      const uint32_t abase = pxa + ((2 * tmi[u] + (mat & 1)) * CR + 8 * (mat >> 1) + mr) * 16;
      const uint32_t bbase = pya + (((mat >> 1) * L.nca + tnj[u]) * CR + 8 * (mat & 1) + mr) * 16;
      const uint32_t ds = static_cast<uint32_t>(L.nca) * CR * 16;  // digit stride
#pragma unroll
      for (int kk = 0; kk < CR / 16; ++kk) {
        uint32_t bf[4][4];  // digits 2 j (registers 0, 1) and 2 j + 1
#pragma unroll
        for (int j = 0; j < 4; ++j) ldsm4_t(bf[j], bbase + kk * 256 + 2 * j * ds);
#pragma unroll
        for (int s = 0; s < 8; ++s) {
          uint32_t af[4];
          ldsm4_t(af, abase + kk * 256 + s * ds);
#pragma unroll
          for (int d = s; d < 8; ++d) {
            const int q = d - s;
            if (d >= 4 && kk >= 2)
              mma_f16(ac2[d - 4], af[0], af[1], af[2], af[3], bf[q / 2][2 * (q & 1)], bf[q / 2][2 * (q & 1) + 1]);
            else
              mma_f16(acc[d], af[0], af[1], af[2], af[3], bf[q / 2][2 * (q & 1)], bf[q / 2][2 * (q & 1) + 1]);
          }
        }
      }
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        int v[8];
#pragma unroll
        for (int d = 0; d < 8; ++d) v[d] = split_int(acc[d][i]) + (d >= 4 ? split_int(ac2[d - 4][i]) : 0);
        const int xe = ex[16 * tmi[u] + g + 8 * (i >> 1)], ye = ey[8 * tnj[u] + 2 * t + (i & 1)];
        int rem;
        const long long o = split_combine(v, rem);
        double r = split_to_double(o + (rem >> 11), xe + ye + 8 - kSplitShift);
        if (xe >= 0x7ff || ye >= 0x7ff) r = __longlong_as_double(0x7ff8000000000000ll);
        sum[u][i] += r;
      }
    }
  };

  double vx[RL][2], vy[SYM ? 1 : RL][2];
  if constexpr (!TM) {
    const int64_t nch = (m + CR - 1) / CR;
    auto fetch = [&](int64_t c) {
      const int64_t r0 = c * CR;
      const int rows = c < nch ? static_cast<int>(m - r0 < CR ? m - r0 : CR) : 0;
      load(X, r0, rows, vx, 0);
      if constexpr (!SYM) load(Yin, r0, rows, vy, 0);
    };
    fetch(blockIdx.x);
    for (int64_t c = blockIdx.x; c < nch; c += gridDim.x) {
      split(vx, pxa, ex, true);
      if constexpr (!SYM) split(vy, pya, ey, false);
      __syncthreads();
      fetch(c + gridDim.x);
      products();
      __syncthreads();
    }
    if (colexp && lane < 4) {
      if (c0 < n && runmax[0] > 0) atomicMax(colexp + c0, runmax[0]);
      if (c0 + 1 < n && runmax[1] > 0) atomicMax(colexp + c0 + 1, runmax[1]);
    }
    double* P = part + static_cast<int64_t>(blockIdx.x) * n * n;
#pragma unroll
    for (int u = 0; u < TW; ++u) {
      if (tmi[u] < 0) continue;
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int r = 16 * tmi[u] + g + 8 * (i >> 1), c = 8 * tnj[u] + 2 * t + (i & 1);
        if (r < n && c < n) {
          if (!SYM) {
            P[r * n + c] = sum[u][i];
          } else if (c >= r) {
            P[r * n + c] = sum[u][i];
            if (c > r) P[c * n + r] = sum[u][i];
          }
        }
      }
    }
  } else {
    // items: tiles; the next chunk's rows are fetched while this one's
    // products run, across tiles
    const int64_t items = p * kt;
    int64_t it = blockIdx.x;
    int off = 0;
    auto rows_of = [&](int64_t i, int64_t& r0, int& tt) {  // rows of tile i (<= 0: none)
      const int64_t blk = i / kt;
      tt = static_cast<int>(i - blk * kt);
      const int64_t rb = m - blk * b < b ? m - blk * b : b;
      const int64_t tr0 = tt == 0 ? 0 : B + static_cast<int64_t>(tt - 1) * bt;
      const int64_t cap = tt == 0 ? B : bt;
      r0 = blk * b + tr0;
      return static_cast<int>(rb - tr0 < cap ? rb - tr0 : cap);
    };
    auto fetch = [&](int64_t i, int o) {
      if (i >= items) return;
      int64_t r0;
      int tt;
      const int cnt = rows_of(i, r0, tt);
      const int rows = cnt - o < CR ? cnt - o : CR;
      load(X, r0 + o, rows, vx, tt == 0 ? o : n);
    };
    int64_t r0;
    int tt;
    while (it < items && rows_of(it, r0, tt) <= 0) it += gridDim.x;
    fetch(it, 0);
    while (it < items) {
      const int cnt = rows_of(it, r0, tt);
      split(vx, pxa, ex, false);
      __syncthreads();
      const int64_t cur = it;
      const bool last = off + CR >= cnt;
      if (last) {
        off = 0;
        it += gridDim.x;
        int64_t rr;
        int t2;
        while (it < items && rows_of(it, rr, t2) <= 0) it += gridDim.x;
      } else {
        off += CR;
      }
      fetch(it, off);
      products();
      if (last) {
        double* P = part + cur * n * n;
#pragma unroll
        for (int u = 0; u < TW; ++u) {
          if (tmi[u] < 0) continue;
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const int r = 16 * tmi[u] + g + 8 * (i >> 1), c = 8 * tnj[u] + 2 * t + (i & 1);
            if (c < n && r < c) P[r * n + c] = sum[u][i];
            sum[u][i] = 0.0;
          }
        }
      }
      __syncthreads();
    }
  }
}

}  // namespace tsqr
