// split.cuh -- binary64 matrix products as exact sums of 8-bit digit products
// on the tensor cores, with the digits formed and recombined in registers
// (mma.sync m16n8k16, binary16 operands, binary32 accumulation).
//
// Splitting (Ozaki, Ogita, Oishi, Rump 2012): a row of the left operand and a
// column of the right one are fixed-point integers against their largest
// exponent, |X| <= 2^62 in 8 balanced digits of 8 bits, X = sum_s d_s 2^(8 (7 -
// s)), -128 <= d_s <= 127 -- exact in binary16.  The products of a diagonal D =
// s + t sum to integers of magnitude at most (D + 1) K 2^14, exact in binary32;
// the diagonals D <= 7 are recombined in 64-bit integers and rounded once to
// binary64.  What is dropped lies 2^-60 (root mean square) below row scale x
// column scale; the fixed point itself rounds at 2^-63 of either scale, so the
// accuracy is normwise: an entry 2^-k of its row's largest keeps 62 - k bits.
// (Rows of 7 digits, 2^-55, for n > 48 doubled the error of small row entries
// and put Step 3 of 3,000 x 64 at 5.5e-16, 4.8e-16 with 8; without diagonal 7
// Cholesky QR at kappa 1e4 came out 1.8 times further from the exact Q.)
//
// Why registers: GB300 has 1.9 binary64 FMAs per clock and SM, against 1024
// binary16 tensor FMAs through mma.sync; 36 digit products per binary64 product
// leave 15 times the binary64 rate.  What bounds these kernels is the integer
// unit (64 lanes a clock) that splits and recombines, so digits go straight
// from the registers that hold an operand's fragment into the product, with no
// pass through shared memory.
#pragma once

#include <cmath>
#include <cstdint>

#include "device.cuh"

namespace tsqr {

// D (16 x 8, binary32) += A (16 x 16) B (16 x 8), binary16 operands.
__device__ __forceinline__ void mma_f16(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3,
                                        uint32_t b0, uint32_t b1) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

// The same with its own addend: D = A B + (c, c, c, c).
__device__ __forceinline__ void mma_f16_c(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3,
                                          uint32_t b0, uint32_t b1, float c) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%10,%10,%10,%10};"
      : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1), "f"(c));
}

constexpr int kExpZero = -100000;  // "exponent" of a zero entry in a maximum
constexpr int kExpBad = 1 << 20;   // ... of a column of M with Inf or NaN

// Biased exponent of x (subnormals count as exponent 1), kExpZero for zero.
__device__ __forceinline__ int split_exp(double x) {
  const uint32_t hi = static_cast<uint32_t>(__double2hiint(x)), lo = static_cast<uint32_t>(__double2loint(x));
  const int e = static_cast<int>((hi >> 20) & 0x7ffu);
  const int f = e > 0 ? e : 1;
  return ((hi << 1) | lo) == 0u ? kExpZero : f;
}

// x 2^(BITS - 1 - (emax - 1023)) rounded to an integer: |x| < 2^(emax - 1022)
// gives |result| <= 2^BITS.  sh = emax - split_exp(x) >= 0 (anything for zero).
template <int BITS>
__device__ __forceinline__ long long split_fixed(double x, int sh) {
  const uint32_t hi = static_cast<uint32_t>(__double2hiint(x)), lo = static_cast<uint32_t>(__double2loint(x));
  const uint32_t mh = (hi & 0xfffffu) | (((hi >> 20) & 0x7ffu) ? 0x100000u : 0u);
  unsigned long long u = (static_cast<unsigned long long>(mh) << 32) | lo;
  u <<= BITS - 52;
  u = sh > 63 ? 0ull : u >> sh;
  u = (u + 1ull) >> 1;
  const long long s = static_cast<long long>(u);
  return static_cast<int>(hi) < 0 ? -s : s;
}

// An accumulator that starts at kSplitMagic holds, in its low bits, the
// integer sum v, |v| <= 2^22: bits = kSplitMagicBits + v.
constexpr float kSplitMagic = 12582912.0f;  // 1.5 2^23
constexpr uint32_t kSplitMagicBits = 0x4B400000u;
__device__ __forceinline__ int split_int(float acc) {
  return static_cast<int>(__float_as_uint(acc) - kSplitMagicBits);
}

// P 2^s rounded to nearest (ties up in magnitude) with integer operations;
// outside the normal range (and for zero) by a call.
#ifdef __CUDA_ARCH__
#define TSQR_SLOW_CALL __noinline__
#else
#define TSQR_SLOW_CALL
#endif
static TSQR_HD TSQR_SLOW_CALL double split_to_double_slow(long long P, int s) {
  return P == 0 ? 0.0 : ldexp(static_cast<double>(P), s);
}
#undef TSQR_SLOW_CALL
TSQR_HD inline double split_to_double(long long P, int s) {
  const unsigned long long up = static_cast<unsigned long long>(P), u = P < 0 ? 0ull - up : up;
  const uint32_t sign = static_cast<uint32_t>(up >> 32) & 0x80000000u;
  const int lz = leading_zeros(u | 1ull);  // at most 63: a shift by 64 has no value
  const unsigned long long w = (u << lz) + 0x400ull;  // bit 63 set; a carry out means 2^64
  // the significand's 53 bits (its hidden bit adds one to the exponent field);
  // a carry out of the rounding leaves w near 0: the exponent takes it
  const uint32_t wl = static_cast<uint32_t>(w), wh = static_cast<uint32_t>(w >> 32);
  const bool carry = wh < 0x80000000u;
  const int e = s - lz + (carry ? 1086 : 1085);  // biased exponent less one
  if (static_cast<uint32_t>(e) > 2044u || u == 0ull) return split_to_double_slow(P, s);
  const uint32_t mh = (carry ? 0x100000u : (wh >> 11));
  const uint32_t ml = funnel_right(wl, wh, 11);
  return from_words(((static_cast<uint32_t>(e) << 20) + mh) | sign, ml);
}

// sum_D v_D 2^(44 - 8 D), D = 0 .. 7: the digit diagonals of a product of two
// operands |X| <= 2^62, in units of 2^68, rounded down, and the rest, 0 <= rem <
// 4096, in units of 2^56.  Sums of at most 64 products: |v_D| <= (D + 1) 2^20
// keeps every step in 32 bits, and the whole below 2^63.
__device__ __forceinline__ long long split_combine(const int (&v)[8], int& rem) {
  const int a = v[1] * 256 + v[2];  // units of 2^28
  const int b = v[3] * 256 + v[4];  // of 2^12
  const int l = v[6] * 256 + v[7];  // of 2^-12
  const int c = v[5] * 16 + (l >> 12);
  rem = l & 4095;
  return static_cast<long long>(v[0]) * (1ll << 44) + static_cast<long long>(a) * (1ll << 28) +
         static_cast<long long>(b) * (1ll << 12) + c;
}
// As P 2^e in units of 2^60: cut to those (e = 0) below 2^55 units of 2^68, else
// rounded to the latter (e = 8), so that P has two bits more than its rounding
// wherever the operands give them.
__device__ __forceinline__ long long split_round(long long o, int rem, int& e) {
  const bool small = static_cast<uint32_t>(static_cast<int>(o >> 32) + 0x800000) < 0x1000000u;
  e = small ? 0 : 8;
  return small ? o * 256 + (rem >> 4) : o + (rem >> 11);
}

// The 8 balanced digits of a pair of fixed-point values (|X|, |Y| <= 2^62).
__device__ __forceinline__ void split_digits(long long X, long long Y, uint32_t (&h)[8]) {
  const unsigned long long bias = 0x8080808080808080ull;
  const unsigned long long x = static_cast<unsigned long long>(X) + bias, y = static_cast<unsigned long long>(Y) + bias;
#pragma unroll
  for (int s = 0; s < 8; ++s) {
    const int byte = 7 - s, jb = byte & 3;
    const uint32_t xa = byte >= 4 ? static_cast<uint32_t>(x >> 32) : static_cast<uint32_t>(x);
    const uint32_t ya = byte >= 4 ? static_cast<uint32_t>(y >> 32) : static_cast<uint32_t>(y);
    const uint32_t v =
        (__byte_perm(xa, ya, static_cast<uint32_t>(jb | ((4 + jb) << 8))) & 0x00ff00ffu) | 0x64006400u;
    asm("sub.rn.f16x2 %0, %1, %2;" : "=r"(h[s]) : "r"(v), "r"(0x64806480u));
  }
}

// Four 8 x 8 binary16 matrices, transposed: matrix i's rows are the 16-byte
// rows at the addresses that lanes 8 i .. 8 i + 7 give; lane (g, t) receives
// the entries (rows 2 t, 2 t + 1; column g).
__device__ __forceinline__ void ldsm4_t(uint32_t (&r)[4], uint32_t addr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(addr)
               : "memory");
}

// ---------------------------------------------------------------------------
// The right operand M (K x N, K = n rows padded to 16 KC, N = n columns padded
// to 8) as digit fragments in shared memory: fragment (j, c, s) of column tile
// j, k step c, digit s at ((j KC + c) 8 + s) 32 + lane, two registers a lane.
// ---------------------------------------------------------------------------
TSQR_HD constexpr int split_kc(int n) { return (n + 15) / 16; }
TSQR_HD constexpr int split_nt(int n) { return (n + 7) / 8; }
TSQR_HD constexpr size_t split_b_bytes(int n) { return static_cast<size_t>(split_nt(n)) * split_kc(n) * 8 * 256; }

// Builds them from row-major M (leading dimension ld, shared or global memory)
// whose row k is taken times 2^kexp[k] (kexp NULL: 1).  cexp[c]: the column's
// exponent.  Whole CTA; ends without a barrier.  `val(k, c)` gives M's entry.
template <class F>
__device__ __forceinline__ void split_build_b(F val, int n, int KC, const int* kexp, int* cexp, uint2* bfrag) {
  const int NT = split_nt(n);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const int g = lane >> 2, t = lane & 3;
  // one warp per column tile: a lane holds column 8 j + g's rows 2 t, 2 t + 1,
  // 2 t + 8, 2 t + 9 of every k step
  for (int j = warp; j < NT; j += nw) {
    const int col = 8 * j + g;
    int em = kExpZero, mx = 0;
    for (int c = 0; c < KC; ++c)
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int k = 16 * c + 2 * t + (i & 1) + 8 * (i >> 1);
        if (k < n && col < n) {
          const int e = split_exp(val(k, col));
          mx = max(mx, e);
          em = max(em, e == kExpZero ? kExpZero : e + (kexp ? kexp[k] : 0));
        }
      }
    em = max(em, __shfl_xor_sync(0xffffffffu, em, 1));
    em = max(em, __shfl_xor_sync(0xffffffffu, em, 2));
    mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, 1));
    mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, 2));
    if (em == kExpZero) em = 0;
    if (t == 0) cexp[col] = mx >= 0x7ff ? kExpBad : em;
    for (int c = 0; c < KC; ++c) {
      long long x[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int k = 16 * c + 2 * t + (i & 1) + 8 * (i >> 1);
        x[i] = 0;
        if (k < n && col < n) {
          const double v = val(k, col);
          const int e = split_exp(v);
          if (e != kExpZero) x[i] = split_fixed<62>(v, em - e - (kexp ? kexp[k] : 0));
        }
      }
      uint32_t h0[8], h1[8];
      split_digits(x[0], x[1], h0);
      split_digits(x[2], x[3], h1);
      uint2* dst = bfrag + static_cast<size_t>(j * KC + c) * 8 * 32 + lane;
#pragma unroll
      for (int s = 0; s < 8; ++s) dst[s * 32] = make_uint2(h0[s], h1[s]);
    }
  }
}

// The left operand: 16 rows of K = 16 KC columns, a lane holding rows g and
// g + 8 at columns 16 c + 2 t, + 1, + 8, + 9 (g = lane / 4, t = lane % 4).
// a[c][s][0..3]: the mma fragment registers of digit s; er[2]: the exponents of
// the two rows (kExpZero for a zero row; a row with Inf or NaN has 0x7ff or
// more when kexp is NULL).  load(r, k): the entry of row r (0..15), column k.
template <int KC, class F>
__device__ __forceinline__ void split_rows(F load, int n, const int* kexp, uint32_t (&a)[KC][8][4], int (&er)[2],
                                           bool (&bad)[2]) {
  const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    double x[KC][4];
    int em = kExpZero;
    int mx = 0;
#pragma unroll
    for (int c = 0; c < KC; ++c)
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int k = 16 * c + 2 * t + (i & 1) + 8 * (i >> 1);
        x[c][i] = load(g + 8 * h, k);
        int e = split_exp(x[c][i]);
        mx = max(mx, e);
        if (kexp) e -= kexp[k];
        em = max(em, e);
      }
    em = max(em, __shfl_xor_sync(0xffffffffu, em, 1));
    em = max(em, __shfl_xor_sync(0xffffffffu, em, 2));
    mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, 1));
    mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, 2));
    er[h] = em;
    bad[h] = mx >= 0x7ff;
#pragma unroll
    for (int c = 0; c < KC; ++c) {
      long long f[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int k = 16 * c + 2 * t + (i & 1) + 8 * (i >> 1);
        int e = static_cast<int>((static_cast<uint32_t>(__double2hiint(x[c][i])) >> 20) & 0x7ffu);
        e = e > 0 ? e : 1;
        if (kexp) e -= kexp[k];
        f[i] = split_fixed<62>(x[c][i], max(em - e, 0));
      }
      uint32_t h0[8], h1[8];
      split_digits(f[0], f[1], h0);
      split_digits(f[2], f[3], h1);
#pragma unroll
      for (int s = 0; s < 8; ++s) {
        a[c][s][h] = h0[s];
        a[c][s][2 + h] = h1[s];
      }
    }
  }
}

// One column tile: o[0], o[1] = row g at columns 2 t, 2 t + 1 of the tile,
// o[2], o[3] = row g + 8.  e0 / e1: er + cexp of the entries' columns.
template <int KC>
__device__ __forceinline__ void split_product(const uint32_t (&a)[KC][8][4], const uint2* bfrag, int lane,
                                              long long (&o)[4], int (&oe)[4]) {
  // diagonals 4 .. 7 of K > 32 in two halves: |v| stays below 2^22
  constexpr int H = KC > 2 ? 2 : 1;
  float acc[8][4], acc2[H > 1 ? 4 : 1][4];
#pragma unroll
  for (int d = 0; d < 8; ++d)
#pragma unroll
    for (int i = 0; i < 4; ++i) acc[d][i] = kSplitMagic;
  if constexpr (H > 1) {
#pragma unroll
    for (int d = 0; d < 4; ++d)
#pragma unroll
      for (int i = 0; i < 4; ++i) acc2[d][i] = kSplitMagic;
  }
#pragma unroll
  for (int c = 0; c < KC; ++c) {
    uint2 b[8];
#pragma unroll
    for (int s = 0; s < 8; ++s) b[s] = bfrag[(c * 8 + s) * 32 + lane];
#pragma unroll
    for (int u = 0; u < 8; ++u)
#pragma unroll
      for (int d = u; d < 8; ++d) {  // digit u of the rows, digit d - u of the columns
        if (H > 1 && d >= 4 && c >= 2)
          mma_f16(acc2[H > 1 ? d - 4 : 0], a[c][u][0], a[c][u][1], a[c][u][2], a[c][u][3], b[d - u].x, b[d - u].y);
        else
          mma_f16(acc[d], a[c][u][0], a[c][u][1], a[c][u][2], a[c][u][3], b[d - u].x, b[d - u].y);
      }
  }
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    int v[8];
#pragma unroll
    for (int d = 0; d < 8; ++d) v[d] = split_int(acc[d][i]);
    if constexpr (H > 1) {
#pragma unroll
      for (int d = 4; d < 8; ++d) v[d] += split_int(acc2[d - 4][i]);
    }
    int rem;
    o[i] = split_combine(v, rem);
    o[i] = split_round(o[i], rem, oe[i]);
  }
}
// value = o 2^(er + cexp + oe - kSplitShift)
constexpr int kSplitShift = 2108;

}  // namespace tsqr
