// panel64.cuh -- Step 1 of direct TSQR (Sec. III-B) for binary64 data:
// Householder QR of one row block per CTA, panels of up to 8 columns factored in
// binary64 and applied to the columns right of them as exact digit products
// on the tensor cores.
//
// Warp q of the CTA's NW = ceil(n / 8) warps owns columns [8 q, 8 q + 8) and
// keeps its 128 rows of the current row tile in shared memory as 62-bit
// fixed-point integers, each column relative to a bound of its whole norm
// (running R and tile): an orthogonal transformation keeps that norm, so the
// scale holds for the tile.  The accuracy is that of the column (normwise): an
// entry 2^-k of its column's norm keeps 62 - k bits.  Per tile the warp applies the block reflectors I - V_p T_p V_p^T
// of the panels p < q as they are published --
//   W = V_p^T A      digits of A (split from the registers) x digits of V_p,
//   W' = T_p^T (W + R's rows of panel p)                     in binary64,
//   A <- A - V_p W'  digits of W' (in the lane that needs them) x digits of V_p,
// the sums recombined straight into the fixed-point tile -- then turns its
// columns into binary64, factors them (eight Householder columns inside one
// warp, no barrier), publishes the digits of V_q and T_q in a ring of
// shared-memory slots, writes V_q to Y and goes on to the next tile while later
// warps are still on this one.
//
// Why: the binary64 unit (1.9 FMAs a clock and SM) was 89 % busy in the
// column-by-column form, which does 2 n^2 flops a row (and 8 % more for the
// running R held in register rows).  Here it does only what lies inside the
// panels, about n / 8 of that; the rest runs on the integer unit and the tensor
// cores, with the digit index packed into the idle halves of the
// fragments.  The running R stays in shared memory: tile t >= 1 factors
// [R; A_t] with vectors [I; V_t].
//
// Measured: Step 1 of 4,000,000 x 64 65.2 -> 20.6 ms plus 3.2 for T's Gram (its
// bytes 0.6; 2 m n^2 binary64 flops would take 27), 3,000,000 x 32 10.96 -> 5.39.
// Bound by the chain of panels a tile runs through: the binary64 unit is 42 %
// busy with conversions, the columns and T_p^T.
#pragma once

#include <cstdint>

#include "device.cuh"
#include "layout.cuh"
#include "qr_kernels.cuh"
#include "split.cuh"

namespace tsqr {

constexpr int kPdCols = 8;
constexpr int kPdRows = 128;  // rows per tile
constexpr int kPdRL = kPdRows / 32;
constexpr int kPdMaxThreads = 512;  // 128 registers a thread
// A slot: 4 planes of 128 16-byte rows, a row the 8 columns' digits 2 j and
// 2 j + 1 as bytes (offset by 128; half the size of binary16 digits, which
// allows twice the slots and so more tiles in flight for four operations a
// register to unpack), 2 I - T (8 x 8) and the 8 column exponents.  It is held from a panel's publication until its last reader, not
// while the panel is factored.
constexpr size_t kPdToff = static_cast<size_t>(kPdRows) * 4 * 16;
constexpr size_t kPdSlotBytes = kPdToff + kPdCols * kPdCols * 8 + 64;
constexpr size_t kPdTileBytes = static_cast<size_t>(kPdRows) * kPdCols * 8;
struct Panel64Smem {
  size_t cnt, slots, tiles, r, wbuf, total;
  TSQR_HD Panel64Smem(int NW, int NS) {
    size_t o = 0;
    cnt = o; o = align_up(o + (2 * static_cast<size_t>(NS) + 1) * 4, 128);
    slots = o; o = align_up(o + NS * kPdSlotBytes, 128);
    tiles = o; o += NW * kPdTileBytes;
    r = o; o += static_cast<size_t>(kPdCols * kPdCols) * 8 * NW * (NW + 1) / 2;  // warp q: 8 (q + 1) rows
    wbuf = o; o += static_cast<size_t>(NW) * 6 * kPdCols * 8;  // two buffers of sums, pivot row, tau, 2 - tau's factors
    total = align_up(o, 16);
  }
};

#if defined(__CUDACC__) && defined(TSQR_PANEL_KERNELS)

// Hand-offs through two counters per ring slot that only grow: the passes
// published and the readers' releases.  (An mbarrier's phase parity cannot
// tell a pass from the one two before it, and warps skip the slots of panels
// right of their own.)  Waits poll with a short sleep and are bounded.
__device__ __forceinline__ uint32_t ld_acquire(const uint32_t* p) {
  uint32_t v;
  asm volatile("ld.acquire.cta.shared::cta.u32 %0, [%1];" : "=r"(v) : "r"(smem_u32(p)) : "memory");
  return v;
}
__device__ __forceinline__ void add_release(uint32_t* p, uint32_t n) {
  asm volatile("red.release.cta.shared::cta.add.u32 [%0], %1;" ::"r"(smem_u32(p)), "r"(n) : "memory");
}
__device__ __forceinline__ bool wait_count(const uint32_t* p, uint32_t want) {
  if (ld_acquire(p) >= want) return true;
  const uint64_t t0 = global_timer_ns();
  while (true) {
#pragma unroll 1
    for (int i = 0; i < 64; ++i) {
      __nanosleep(64);
      if (ld_acquire(p) >= want) return true;
    }
    if (global_timer_ns() - t0 > kWaitLimitNs) return false;
  }
}
// A position in the ring of slots: slot index and its pass (0, 1, ..).
struct RingPos {
  int slot;
  uint32_t pass;
  __device__ void advance(int k, int ns) {
    slot += k;
    while (slot >= ns) {
      slot -= ns;
      ++pass;
    }
  }
};

__device__ __forceinline__ void ldsm4(uint32_t (&r)[4], uint32_t addr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(addr)
               : "memory");
}

// A pair of values' digits 2 j and 2 j + 1 (bytes a, a', b, b' offset by 128)
// as binary16 pairs.
__device__ __forceinline__ void unpack_digits(uint32_t r, uint32_t& h0, uint32_t& h1) {
  const uint32_t v0 = __byte_perm(r, 0x64646464u, 0x4240), v1 = __byte_perm(r, 0x64646464u, 0x4341);
  asm("sub.rn.f16x2 %0, %1, %2;" : "=r"(h0) : "r"(v0), "r"(0x64806480u));
  asm("sub.rn.f16x2 %0, %1, %2;" : "=r"(h1) : "r"(v1), "r"(0x64806480u));
}

__device__ __forceinline__ int biased_exp(double x) {  // subnormals and zero: 1
  const int e = (__double2hiint(x) >> 20) & 0x7ff;
  return e > 0 ? e : 1;
}

// The tile's index of (row, column): 64-byte rows, two to a 128-byte line, the
// halves and columns exchanged so that both walks are free of bank conflicts:
// eight columns of rows 2 t (the fragments') and one column of 32 rows.
__device__ __forceinline__ int tile_at(int r, int c) {
  return (r >> 1) * 16 + (((r ^ (r >> 1)) & 1) << 3) + (c ^ ((r >> 2) & 7));
}

// x 2^(1085 - sc) truncated to an integer (|x| < 2^(sc - 1023): below 2^62);
// with sc + 1 in place of sc, split_fixed<62> without its rounding, which is a
// unit of 2^-62.
__device__ __forceinline__ long long fixed_of(double x, int sc) {
  const uint32_t hi = static_cast<uint32_t>(__double2hiint(x)), lo = static_cast<uint32_t>(__double2loint(x));
  const int e = static_cast<int>((hi >> 20) & 0x7ffu);
  const uint32_t mh = (hi & 0xfffffu) | (e > 0 ? 0x100000u : 0u);
  const int sh = min(sc - (e > 0 ? e : 1), 63);
  uint32_t ah = __funnelshift_l(lo, mh, 10), al = lo << 10;
  if (sh >= 32) {
    al = ah;
    ah = 0u;
  }
  al = __funnelshift_r(al, ah, sh);
  ah >>= sh & 31;
  const long long s = static_cast<long long>((static_cast<unsigned long long>(ah) << 32) | al);
  return static_cast<int>(hi) < 0 ? -s : s;
}

// One column of the panel factorisation (rows lane + 32 i in a[i]).
// rbuf: the pivot row (tile 0) is exchanged there, then tau and the factors of 2 -
// tau; sbuf: the sums.
template <int J>
__device__ __forceinline__ void panel64_column(double (&a)[kPdRL][kPdCols], double* Rq, double* sbuf, double* rbuf,
                                               int j0, int nb, bool first, int lane) {
  const int r = j0 + J;
  const double* prow = Rq + r * kPdCols;
  if (first) {
    const int ir = r >> 5;
    if (lane == (r & 31)) {
#pragma unroll
      for (int i = 0; i < kPdRL; ++i)
        if (i == ir) {
#pragma unroll
          for (int c = J; c < kPdCols; ++c) {
            rbuf[c] = a[i][c];
            a[i][c] = 0.0;  // the row leaves the tile: it is R's from here on
          }
        }
    }
    __syncwarp();
    prow = rbuf;
  }
  double* dst = sbuf + (J & 1) * kPdCols;
  {
    double s[kPdCols - J];
#pragma unroll
    for (int c = J; c < kPdCols; ++c) {
      s[c - J] = 0.0;
      if (c < nb) {  // (warp-uniform: a narrow panel's padding costs nothing)
        double acc = a[0][J] * a[0][c];
#pragma unroll
        for (int i = 1; i < kPdRL; ++i) acc = fma(a[i][J], a[i][c], acc);
        s[c - J] = acc;
      }
    }
    TransposeReduce<kPdCols - J, 16>::run(s, lane, 0, kPdCols - J, dst + J);
  }
  __syncwarp();
  const double alpha = prow[J], sj = dst[J];
  const Reflector<double> f = make_reflector64(fma(alpha, alpha, sj), alpha);
  const double ps = sj * f.scal;
  if (lane == 0) {  // tau and the factors of 2 - tau (panel64_comp)
    rbuf[kPdCols + J] = f.tau;
    rbuf[2 * kPdCols + J] = f.ident ? 2.0 : ps;
    rbuf[3 * kPdCols + J] = f.ident ? -1.0 : f.ib;
  }
  // lane c: column c's row of R and its coefficient of x.  r' = (alpha r + s) /
  // beta, from tile 1 on as -r + (s + (alpha + beta) r) / beta with alpha + beta
  // = -s_J / (alpha - beta): there alpha is close to -beta, so the correction is
  // small and the running R takes one rounding a tile (in tile 0 alpha is one
  // entry, and that form would cancel)
  double dl = 0.0, rn = 0.0;
  const bool trail = lane > J && lane < nb;
  if (trail) {
    const double rc = prow[lane];
    rn = f.ident ? rc : first ? fma(alpha, rc, dst[lane]) * f.ib : fma(fma(-ps, rc, dst[lane]), f.ib, -rc);
    dl = (rn - rc) * f.scal;
  }
  __syncwarp();  // the pivot row has been read
  if (trail) Rq[r * kPdCols + lane] = rn;
  else if (lane == J) Rq[r * kPdCols + J] = f.beta;
#pragma unroll
  for (int c = J + 1; c < kPdCols; ++c) {
    const double d = __shfl_sync(0xffffffffu, dl, c);
    if (c < nb) {
#pragma unroll
      for (int i = 0; i < kPdRL; ++i) a[i][c] = fma(d, a[i][J], a[i][c]);
    }
  }
#pragma unroll
  for (int i = 0; i < kPdRL; ++i) a[i][J] *= f.scal;
  if (first) {
    const int ir = r >> 5;
    if (lane == (r & 31)) {
#pragma unroll
      for (int i = 0; i < kPdRL; ++i)
        if (i == ir) a[i][J] = 1.0;
    }
  }
}

// Columns J .. nb - 1 (the padding columns of a last panel are zero: they give
// zero vectors and tau = 0).
template <int J>
__device__ __forceinline__ void panel64_factor(double (&a)[kPdRL][kPdCols], double* Rq, double* sbuf, double* rbuf,
                                               int j0, int nb, bool first, int lane) {
  if constexpr (J < kPdCols) {
    if (J < nb) panel64_column<J>(a, Rq, sbuf, rbuf, j0, nb, first, lane);
    panel64_factor<J + 1>(a, Rq, sbuf, rbuf, j0, nb, first, lane);
  }
}

// 2 - tau of the panel's columns, lane c for column c (each of the unit's
// instructions takes a warp 64 clocks, so one for the eight): s_J / (root
// (|alpha| + root)) with a relative error of its own -- taken from the rounded
// tau it errs by tau's rounding, which a block's every tile adds to Q.  (Nor tau
// as 2 minus this: d r shares d's rounding with scal = 1 / d; Q's error at 2,000 x 8
// rose by a tenth.)  Into rbuf's third row.
__device__ __forceinline__ void panel64_comp(double* rbuf, int lane) {
  if (lane < kPdCols) rbuf[2 * kPdCols + lane] = -(rbuf[2 * kPdCols + lane] * rbuf[3 * kPdCols + lane]);
  __syncwarp();
}

// ---------------------------------------------------------------------------
// grid = p row blocks of b rows, tiles of 128 rows (kt T slots a block).
// Outputs as k_local_qr without Gram dot products: Y (the vectors; NULL: R
// only), R_i (raw signs), tau_j on the T slots' diagonals (Tst, with Y).
// Every panel but the last is published; a slot is released by NW arrivals: the
// warps right of its panel, and its owner for the rest.
// The loops over a tile's rows stay rolled: with the tile in registers they
// are unrolled whole, and the 16 warps, each at another place, then missed the
// instruction cache on every second fetch.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(kPdMaxThreads, 1)
    k_panel_qr_f64(const double* __restrict__ A, int64_t m, int n, int b, int kt, int NW, int NS, uint64_t order,
                   int sms, double* Y, double* __restrict__ Rst, double* __restrict__ Tst, int32_t* status) {
  constexpr int TR = kPdRows, RL = kPdRL;
  extern __shared__ __align__(128) unsigned char smem[];
  const Panel64Smem L(NW, NS);
  uint32_t* full = reinterpret_cast<uint32_t*>(smem + L.cnt);  // passes published
  uint32_t* freed = full + NS;                                  // releases, NW per pass
  uint32_t* bad = full + 2 * NS;  // n less the first column that met Inf or NaN (0: none)
  const int lane = threadIdx.x & 31;
  // Panels differ in work and warp w sits on sub-partition w mod 4 in every CTA:
  // order deals them evenly (choose_panel); with one warp a sub-partition the
  // start moves with the CTA instead, an SM's first CTAs being a device's SM
  // count apart.  (The moving start at every n: Step 1 of 2,000,000 x 50
  // 10.06 ms, 7.69 dealt evenly; x 40 5.76 and 4.79; 4,000,000 x 64 21.8 and
  // 20.9; 1,000,000 x 72 7.79 and 6.60.)
  const unsigned w = threadIdx.x / 32;
  const int q = NW > 4 ? static_cast<int>((order >> (4 * w)) & 15u)
                       : static_cast<int>((w + blockIdx.x + blockIdx.x / static_cast<unsigned>(sms)) %
                                         static_cast<unsigned>(NW));
  const int g = lane >> 2, t4 = lane & 3;
  const int64_t row0 = static_cast<int64_t>(blockIdx.x) * b;
  const int rows = static_cast<int>(m - row0 < b ? m - row0 : b);
  const int ntiles = row_tiles(rows, TR, TR);
  for (int s = threadIdx.x; s < 2 * NS + 1; s += blockDim.x) full[s] = 0;
  // R starts as zero: its entries below the diagonal and of padding columns
  // are read (as part of a column's norm) but never written
  for (size_t s = L.r / 8 + threadIdx.x; s < L.wbuf / 8; s += blockDim.x) reinterpret_cast<double*>(smem)[s] = 0.0;
  __syncthreads();

  const int j0 = kPdCols * q, nb = n - j0 < kPdCols ? n - j0 : kPdCols;
  double* Rq = reinterpret_cast<double*>(smem + L.r) + kPdCols * kPdCols * q * (q + 1) / 2;
  double* sbuf = reinterpret_cast<double*>(smem + L.wbuf) + static_cast<size_t>(q) * 6 * kPdCols;
  double* rbuf = sbuf + 2 * kPdCols;
  long long* X = reinterpret_cast<long long*>(smem + L.tiles + static_cast<size_t>(q) * kPdTileBytes);
  double* Xd = reinterpret_cast<double*>(X);
  const bool own = g < nb;  // this lane's column j0 + g is one, where lanes go by fragments
  RingPos pos{0, 0};
  bool nonfinite = false;
  for (int t = 0; t < ntiles; ++t) {
    const int tr0 = t * TR;
    const int cnt = rows - tr0 < TR ? rows - tr0 : TR;
    const bool first = t == 0;
    // ---- the tile's columns (lane: rows 8 i + 2 t4, + 1 of column g)
    int sc;  // |column| < 2^(sc - 1023), running R included
    {
      const double* p0 = A + (row0 + tr0 + 2 * t4) * n + j0 + g;
      int em = 1;
#pragma unroll 8
      for (int i = 0; i < TR / 8; ++i)
#pragma unroll
        for (int u = 0; u < 2; ++u) {
          double v = 0.0;
          if (own && 8 * i + 2 * t4 + u < cnt) v = p0[static_cast<int64_t>(8 * i + u) * n];
          Xd[tile_at(8 * i + 2 * t4 + u, g)] = v;
          em = max(em, (__double2hiint(v) >> 20) & 0x7ff);
        }
      // the column of R: its largest exponent, then its squared norm in units
      // of 4^(e0 - 20) with 21-bit significands
      int er = 1;
      if (!first)
        for (int i = t4; i < j0 + nb; i += 4) er = max(er, biased_exp(Rq[i * kPdCols + g]));
      int e0 = max(em, er);
      e0 = max(e0, __shfl_xor_sync(0xffffffffu, e0, 1));
      e0 = max(e0, __shfl_xor_sync(0xffffffffu, e0, 2));
      em = max(em, __shfl_xor_sync(0xffffffffu, em, 1));
      em = max(em, __shfl_xor_sync(0xffffffffu, em, 2));
      float s2 = 0.0f;
      if (!first)
        for (int i = t4; i < j0 + nb; i += 4) {
          const double rv = Rq[i * kPdCols + g];
          const int sh = e0 - biased_exp(rv);
          const int mh = ((__double2hiint(rv) & 0xfffff) | 0x100000) + 1;
          const float fv = sh > 24 ? 1.0f : static_cast<float>((mh >> sh) + 1);
          s2 = fmaf(fv, fv, s2);
        }
      s2 += __shfl_xor_sync(0xffffffffu, s2, 1);
      s2 += __shfl_xor_sync(0xffffffffu, s2, 2);
      // the tile: at most TR entries below 2^(em + 1)
      const int d = e0 - em;
      const float am = d > 24 ? 4.0f : static_cast<float>((1 << 21) >> d) + 1.0f;
      s2 = fmaf(am * am, static_cast<float>(TR), s2) * 1.001f;
      // norm < 2^((exponent of s2 + 1) / 2) in units of 2^(e0 - 20)
      const int e2 = static_cast<int>(__float_as_uint(s2) >> 23) - 127;
      sc = e0 - 20 + ((e2 + 2) >> 1);
      if (e0 >= 0x7ff) nonfinite = true;
      if (q > 0) {  // panel 0 is never fixed point
#pragma unroll 2
        for (int i = 0; i < TR / 8; ++i)
#pragma unroll
          for (int u = 0; u < 2; ++u) {
            const int k = tile_at(8 * i + 2 * t4 + u, g);
            X[k] = fixed_of(Xd[k], sc);
          }
      }
    }
    // ---- block reflectors of the panels to the left
    for (int p = 0; p < q; ++p) {
      if (!wait_count(full + pos.slot, pos.pass + 1)) {
        if (lane == 0) set_status(status, TSQR_ERR_TIMEOUT);
        return;
      }
      const unsigned char* sl = smem + L.slots + static_cast<size_t>(pos.slot) * kPdSlotBytes;
      const uint32_t va = smem_u32(sl);
      const double* T = reinterpret_cast<const double*>(sl + kPdToff);
      const int* ev = reinterpret_cast<const int*>(T + kPdCols * kPdCols);
      const int jp = kPdCols * p;
      double w0, w1;  // W' at reflectors 2 t4, 2 t4 + 1, column g
      {
        // W^T = A^T V: A's digits s and s + 1 in the fragment's two row halves
        float acc[8][4];
#pragma unroll
        for (int d = 0; d < 8; ++d)
#pragma unroll
          for (int i = 0; i < 4; ++i) acc[d][i] = 0.0f;
        // lanes 8 k .. 8 k + 7 address matrix k: rows 0-7, 8-15 of plane 2 j, then of 2 j + 1
        const uint32_t vl = va + ((lane >> 4) * TR + ((lane >> 3) & 1) * 8 + (lane & 7)) * 16;
#pragma unroll 1
        for (int i = 0; i < TR / 16; ++i) {
          uint32_t v0[8], v1[8];  // V's digits, rows 16 i + 2 t4 (+ 1) and 8 further
#pragma unroll
          for (int j = 0; j < 2; ++j) {
            uint32_t pk[4];
            ldsm4_t(pk, vl + (2 * j * TR + 16 * i) * 16);
            unpack_digits(pk[0], v0[4 * j], v0[4 * j + 1]);
            unpack_digits(pk[1], v1[4 * j], v1[4 * j + 1]);
            unpack_digits(pk[2], v0[4 * j + 2], v0[4 * j + 3]);
            unpack_digits(pk[3], v1[4 * j + 2], v1[4 * j + 3]);
          }
          uint32_t h0[8], h1[8];
          const int r = 16 * i + 2 * t4;
          split_digits(X[tile_at(r, g)], X[tile_at(r + 1, g)], h0);
          split_digits(X[tile_at(r + 8, g)], X[tile_at(r + 9, g)], h1);
#pragma unroll
          for (int bq = 0; bq < 8; ++bq)
#pragma unroll
            for (int s = 0; s + bq < 8; s += 2)
              mma_f16(acc[s + bq], h0[s], h0[s + 1], h1[s], h1[s + 1], v0[bq], v1[bq]);
        }
        double w[2];
#pragma unroll
        for (int u = 0; u < 2; ++u) {
          long long r[2] = {0, 0};  // diagonals 0 .. 3 in units of 2^88, 4 .. 7 of 2^56
#pragma unroll
          for (int d = 0; d < 8; ++d) {
            const int v = __float2int_rn(acc[d][u]) + (d > 0 ? __float2int_rn(acc[d > 0 ? d - 1 : 0][2 + u]) : 0);
            r[d / 4] += static_cast<long long>(v) << (24 - 8 * (d & 3));
          }
          const int s = sc + ev[2 * t4 + u] - 2169;
          w[u] = split_to_double(r[0], s + 88) + split_to_double(r[1], s + 56);
        }
        // W' = T^T Z, Z = W + R's rows, within the column's four lanes: with E =
        // 2 I - T (small in a block's later tiles, whose tau are close to 2) it
        // is 2 Z - E^T Z, and R - W' = E^T Z - 2 W - R takes one rounding of R
        double r0 = 0.0, r1 = 0.0;
        double* rp = Rq + (jp + 2 * t4) * kPdCols + g;
        const double wa = w[0], wc = w[1];
        if (!first) {
          r0 = rp[0];
          r1 = rp[kPdCols];
          w[0] += r0;
          w[1] += r1;
        }
        w0 = w1 = 0.0;  // E^T Z
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const double a0 = __shfl_sync(0xffffffffu, w[0], (lane & ~3) | i);
          const double a1 = __shfl_sync(0xffffffffu, w[1], (lane & ~3) | i);
          const double2 ta = *reinterpret_cast<const double2*>(T + (2 * i) * kPdCols + 2 * t4);
          const double2 tb = *reinterpret_cast<const double2*>(T + (2 * i + 1) * kPdCols + 2 * t4);
          w0 = fma(ta.x, a0, w0);
          w1 = fma(ta.y, a0, w1);
          w0 = fma(tb.x, a1, w0);
          w1 = fma(tb.y, a1, w1);
        }
        if (!first) {
          rp[0] = fma(-2.0, wa, w0) - r0;
          rp[kPdCols] = fma(-2.0, wc, w1) - r1;
        }
        w0 = fma(2.0, w[0], -w0);
        w1 = fma(2.0, w[1], -w1);
      }
      // A -= V W': the digits of -W' 2^(ev) relative to the column's scale.  W'_j =
      // tau_j v_j^T b with b the column after j reflectors, so |W'_j| <= 2 ||b|| / ||v_j||
      // <= 2 norms, and V's entries are at most 1: the shifts are not negative (but
      // for a column with Inf or NaN, which is NaN in the end).
      {
        const int s0 = sc + 1023 - biased_exp(w0) - ev[2 * t4], s1 = sc + 1023 - biased_exp(w1) - ev[2 * t4 + 1];
        uint32_t h[8];
        split_digits(split_fixed<62>(-w0, max(s0, 0)), split_fixed<62>(-w1, max(s1, 0)), h);
        // matrices 0 .. 3: the eight rows of the four planes
        const uint32_t vl = va + ((lane >> 3) * TR + (lane & 7)) * 16;
#pragma unroll 2
        for (int i = 0; i < TR / 8; ++i) {
          uint32_t pk[4], vd[8];
          ldsm4(pk, vl + 8 * i * 16);
#pragma unroll
          for (int j = 0; j < 4; ++j) unpack_digits(pk[j], vd[2 * j], vd[2 * j + 1]);
          float acc[5][4];
          // k 0-7: digit v of V against digits s, s + 1 of W'; k 8-15: digit
          // v + 1 against s - 1, s.  Diagonals 0 .. 8 (dropping the last too
          // would cost 10 units of the column's fixed point a panel)
#pragma unroll
          for (int v = 0; v < 8; v += 2)
#pragma unroll
            for (int s = 0; s + v <= 8; s += 2) {
              const uint32_t a0 = s < 8 ? h[s & 7] : 0u, a1 = s < 7 ? h[(s + 1) & 7] : 0u;
              const uint32_t a2 = s > 0 ? h[(s + 7) & 7] : 0u;
              if (v == 0) mma_f16_c(acc[s / 2], a0, a1, a2, a0, vd[0], vd[1], kSplitMagic);
              else mma_f16(acc[(s + v) / 2], a0, a1, a2, a0, vd[v], vd[v + 1]);
            }
          // sum_D v_D 2^(52 - 8 D) from the accumulators' bits (kSplitMagicBits
          // + v_D): pairs in 32 bits, the constants taken out once each
#pragma unroll
          for (int u = 0; u < 2; ++u) {
            auto bits = [&](int d) { return __float_as_uint(acc[d / 2][2 * (d & 1) + u]); };
            constexpr uint32_t K2 = kSplitMagicBits * 257u, K3 = kSplitMagicBits * 65793u;
            const uint32_t hi = (bits(0) * 256u + bits(1)) * 256u + bits(2) - K3;  // units of 2^36
            const int a = static_cast<int>(bits(3) * 256u + bits(4) - K2);
            const int bb = static_cast<int>(bits(5) * 256u + bits(6) - K2);
            const int c = static_cast<int>(bits(7) * 256u + bits(8) - (K2 - 2048u)) >> 12;
            long long r = static_cast<long long>(a) * 1048576 + static_cast<long long>(bb) * 16 + c;
            r += static_cast<long long>(static_cast<unsigned long long>(hi) << 36);
            X[tile_at(8 * i + 2 * t4 + u, g)] += r;
          }
        }
      }
      __syncwarp();
      if (lane == 0) add_release(freed + pos.slot, 1);
      if (first) {  // tile 0: the panel's pivot rows leave the tile
#pragma unroll
        for (int u = 0; u < 2; ++u) {
          const int r = jp + 2 * t4 + u, k = tile_at(r, g);
          Rq[r * kPdCols + g] = split_to_double(X[k], sc - 1085);
          X[k] = 0;
        }
        __syncwarp();
      }
      pos.advance(1, NS);
    }
    // ---- own panel: fixed point -> binary64, then rows lane + 32 i.  A column that
    // met Inf or NaN has no fixed point: NaN, so that its vector, its tau and with
    // them the block's Q become NaN (a caller that reads Q alone sees it)
    if (q > 0) {
#pragma unroll 2
      for (int i = 0; i < TR / 8; ++i)
#pragma unroll
        for (int u = 0; u < 2; ++u) {
          const int k = tile_at(8 * i + 2 * t4 + u, g);
          Xd[k] = nonfinite ? __longlong_as_double(0x7ff8000000000000ll) : split_to_double(X[k], sc - 1085);
        }
    }
    __syncwarp();
    double a[RL][kPdCols];
#pragma unroll
    for (int i = 0; i < RL; ++i)
#pragma unroll
      for (int c = 0; c < kPdCols; ++c) a[i][c] = Xd[tile_at(lane + 32 * i, c)];
    panel64_factor<0>(a, Rq, sbuf, rbuf, j0, nb, first, lane);
    __syncwarp();
    panel64_comp(rbuf, lane);
    // ---- V through the tile: digits (62-bit fixed point per column) and Y
#pragma unroll
    for (int i = 0; i < RL; ++i)
#pragma unroll
      for (int c = 0; c < kPdCols; ++c) Xd[tile_at(lane + 32 * i, c)] = a[i][c];
    if (q + 1 < NW) {
      // publish, once the slot's previous panel has been read by all
      int e[kPdCols];
#pragma unroll
      for (int c = 0; c < kPdCols; ++c) {
        uint32_t mx = 0;
#pragma unroll
        for (int i = 0; i < RL; ++i) mx = max(mx, static_cast<uint32_t>(__double2hiint(a[i][c])) & 0x7fffffffu);
        e[c] = max(1, static_cast<int>(__reduce_max_sync(0xffffffffu, mx) >> 20));
      }
      if (!wait_count(freed + pos.slot, pos.pass * NW)) {
        if (lane == 0) set_status(status, TSQR_ERR_TIMEOUT);
        return;
      }
      unsigned char* sl = smem + L.slots + static_cast<size_t>(pos.slot) * kPdSlotBytes;
      double* T = reinterpret_cast<double*>(sl + kPdToff);
      int* ev = reinterpret_cast<int*>(T + kPdCols * kPdCols);
#pragma unroll
      for (int c = 0; c < kPdCols; ++c)
        if (lane == c) ev[c] = e[c];
      __syncwarp();
#pragma unroll 1
      for (int i = 0; i < RL; ++i) {
        const int r = lane + 32 * i;
        uint32_t h[4][4];  // plane j, columns 2 c and 2 c + 1
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          constexpr unsigned long long bias = 0x8080808080808080ull;
          const unsigned long long x = static_cast<unsigned long long>(fixed_of(Xd[tile_at(r, 2 * c)], e[2 * c] + 1)) + bias;
          const unsigned long long y =
              static_cast<unsigned long long>(fixed_of(Xd[tile_at(r, 2 * c + 1)], e[2 * c + 1] + 1)) + bias;
          const uint32_t xh = static_cast<uint32_t>(x >> 32), yh = static_cast<uint32_t>(y >> 32);
          h[0][c] = __byte_perm(xh, yh, 0x6723);
          h[1][c] = __byte_perm(xh, yh, 0x4501);
          h[2][c] = __byte_perm(static_cast<uint32_t>(x), static_cast<uint32_t>(y), 0x6723);
          h[3][c] = __byte_perm(static_cast<uint32_t>(x), static_cast<uint32_t>(y), 0x4501);
        }
#pragma unroll
        for (int j = 0; j < 4; ++j)
          *reinterpret_cast<uint4*>(sl + static_cast<size_t>(j * TR + r) * 16) =
              make_uint4(h[j][0], h[j][1], h[j][2], h[j][3]);
      }
      __syncwarp();
      {
        float acc[8][4];
#pragma unroll
        for (int d = 0; d < 8; ++d)
#pragma unroll
          for (int i = 0; i < 4; ++i) acc[d][i] = 0.0f;
        const uint32_t vl = smem_u32(sl) + ((lane >> 4) * TR + ((lane >> 3) & 1) * 8 + (lane & 7)) * 16;
#pragma unroll 1
        for (int i = 0; i < TR / 16; ++i) {
          uint32_t v0[8], v1[8];
#pragma unroll
          for (int j = 0; j < 2; ++j) {
            uint32_t pk[4];
            ldsm4_t(pk, vl + (2 * j * TR + 16 * i) * 16);
            unpack_digits(pk[0], v0[4 * j], v0[4 * j + 1]);
            unpack_digits(pk[1], v1[4 * j], v1[4 * j + 1]);
            unpack_digits(pk[2], v0[4 * j + 2], v0[4 * j + 3]);
            unpack_digits(pk[3], v1[4 * j + 2], v1[4 * j + 3]);
          }
#pragma unroll
          for (int bq = 0; bq < 8; ++bq)
#pragma unroll
            for (int s = 0; s + bq < 8; s += 2)
              mma_f16(acc[s + bq], v0[s], v0[s + 1], v1[s], v1[s + 1], v0[bq], v1[bq]);
        }
        // G(g, 2 t4 + u) into T's place, then T row by row: lane i < 8 forms
        // T(i, J) = -tau_J sum_l T(i, l) G(l, J)
#pragma unroll
        for (int u = 0; u < 2; ++u) {
          long long r[2] = {0, 0};  // diagonals 0 .. 3 in units of 2^88, 4 .. 7 of 2^56
#pragma unroll
          for (int d = 0; d < 8; ++d) {
            const int v = __float2int_rn(acc[d][u]) + (d > 0 ? __float2int_rn(acc[d > 0 ? d - 1 : 0][2 + u]) : 0);
            r[d / 4] += static_cast<long long>(v) << (24 - 8 * (d & 3));
          }
          const int c = 2 * t4 + u, s = ev[g] + ev[c] - 2168;
          T[g * kPdCols + c] = split_to_double(r[0], s + 88) + split_to_double(r[1], s + 56);
        }
      }
      __syncwarp();
      double tr[kPdCols];
#pragma unroll
      for (int J = 0; J < kPdCols; ++J) {
        double s = 0.0;
#pragma unroll
        for (int l = 0; l < J; ++l) s = fma(tr[l], T[l * kPdCols + J], s);
        tr[J] = lane < J ? -rbuf[kPdCols + J] * s : (lane == J ? rbuf[kPdCols + J] : 0.0);
      }
      __syncwarp();
      if (lane < kPdCols) {
#pragma unroll
        for (int c = 0; c < kPdCols; ++c) T[lane * kPdCols + c] = lane == c ? rbuf[2 * kPdCols + c] : -tr[c];  // E = 2 I - T
      }
      __syncwarp();
      if (lane == 0) {
        add_release(full + pos.slot, 1);
        add_release(freed + pos.slot, q + 1);  // the warps right of it arrive NW - 1 - q times
      }
      pos.advance(NW - 1 - q, NS);
    }
    __syncwarp();
    if (Y) {
      // eight lanes a row
      double* yg = Y + (row0 + tr0) * n + j0 + (lane & 7);
      if ((lane & 7) < nb) {
#pragma unroll 4
        for (int r = lane >> 3; r < cnt; r += 4) yg[static_cast<int64_t>(r) * n] = Xd[tile_at(r, lane & 7)];
      }
      double* Tg = Tst + (static_cast<int64_t>(blockIdx.x) * kt + t) * n * n;
#pragma unroll
      for (int c = 0; c < kPdCols; ++c)
        if (lane == c && c < nb) {
          Tg[static_cast<int64_t>(j0 + c) * (n + 1)] = rbuf[kPdCols + c];
          Tg[comp_at(j0 + c, n)] = rbuf[2 * kPdCols + c];
        }
      __syncwarp();
    }
  }
  // ---- R_i (raw signs); NaN from the first column that met Inf or NaN on
  if (nonfinite && t4 == 0) atomicMax(bad, static_cast<unsigned>(n - (j0 + g)));
  __syncthreads();
  const int first_bad = n - static_cast<int>(*bad);
  double* Rg = Rst + static_cast<int64_t>(blockIdx.x) * n * n;
  for (int e = lane; e < n * kPdCols; e += 32) {
    const int r = e / kPdCols, c = e - r * kPdCols;
    if (c < nb) {
      double v = (j0 + c >= r && r < rows) ? Rq[r * kPdCols + c] : 0.0;
      if (j0 + c >= first_bad) v = __longlong_as_double(0x7ff8000000000000ll);
      Rg[static_cast<int64_t>(r) * n + j0 + c] = v;
    }
  }
}

#endif  // TSQR_PANEL_KERNELS

}  // namespace tsqr
