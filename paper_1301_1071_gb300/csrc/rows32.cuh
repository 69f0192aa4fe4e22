// rows32.cuh -- rows times an n x n matrix for binary32 data on the FMA units:
// out = X M1 + Y M2 (Q = A R^-1, the adjoint) and the native Step 3.
//
// A CTA takes 128 rows; a thread 8 rows x 8 columns of the output in packed
// registers, so that per k step it reads 8 values of the rows (16 bytes at a
// time) and 8 of the matrix for 64 FMAs.  k_rowmul and k_form_q gave a thread 24
// or 12 rows x 5 or 8 columns with one 4-byte shared load per row and k: 18 % of
// the FMA rate at n = 64.  Row tiles arrive by cp.async one tile ahead, in rows
// padded to ld = 4 mod 8 floats (conflict-free 16-byte reads of adjacent rows).
// 4,000,000 x 64: out = X M1 + Y M2 4.27 -> 1.80 ms (bound by the FMA pipe:
// 32.8 G FMA at 19,456 a clock 0.85 ms, the 3.07 GB 0.46), Step 3 5.04 -> 1.51 ms.
#pragma once

#include <cstdint>

#include "device.cuh"
#include "layout.cuh"

namespace tsqr {

constexpr int kR32Rows = 128;
constexpr int kR32Ty = 16;  // row groups; a thread's rows are ty + 16 i
TSQR_HD constexpr int r32_tx(int n) { return (n + 7) / 8; }
TSQR_HD constexpr int r32_kp(int n) { return (n + 3) / 4 * 4; }
TSQR_HD constexpr int r32_ld(int n) { return r32_kp(n) % 8 == 4 ? r32_kp(n) : r32_kp(n) + 4; }
TSQR_HD constexpr int r32_np(int n) { return 8 * r32_tx(n); }
TSQR_HD constexpr size_t r32_mat(int n) { return static_cast<size_t>(r32_kp(n)) * r32_np(n) * 4; }
TSQR_HD constexpr size_t r32_tile(int n) { return static_cast<size_t>(kR32Rows) * r32_ld(n) * 4; }

#if defined(__CUDACC__) && defined(TSQR_ROWS32_KERNELS)

using f32x2 = unsigned long long;
__device__ __forceinline__ f32x2 pack2(float lo, float hi) {
  f32x2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ float2 unpack2(f32x2 v) {
  float2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
  return r;
}
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
  f32x2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
__device__ __forceinline__ void cp_async_16(void* dst_smem, const void* src_gmem) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(dst_smem)), "l"(src_gmem) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait_1() { asm volatile("cp.async.wait_group 1;" ::: "memory"); }

// Starts the copy of `rows` rows of n floats at g into a tile (16, 8 or 4 bytes
// a copy, as the rows' alignment allows).
__device__ __forceinline__ void r32_load(float* tile, const float* g, int rows, int n, int ld) {
  const int w = ((n & 3) == 0 && (reinterpret_cast<uintptr_t>(g) & 15) == 0)  ? 4
                : ((n & 1) == 0 && (reinterpret_cast<uintptr_t>(g) & 7) == 0) ? 2
                                                                              : 1;
  const int per = n / w, total = rows * per;  // copy i: row i / per, stepped without division
  const int dr = blockDim.x / per, dc = blockDim.x - dr * per;
  int r = threadIdx.x / per, c = threadIdx.x - r * per;
  for (int i = threadIdx.x; i < total; i += blockDim.x) {
    float* d = tile + r * ld + c * w;
    const float* s = g + i * w;
    if (w == 4) cp_async_16(d, s);
    else if (w == 2) cp_async_8(d, s);
    else cp_async_4(d, s);
    r += dr;
    c += dc;
    if (c >= per) {
      c -= per;
      ++r;
    }
  }
}

using R32Acc = f32x2[8][4];  // row ty + 16 i, columns 8 tx + 2 c, + 1

// acc += tile rows x mat (KP x NP row-major, zero-padded rows).
__device__ __forceinline__ void r32_product(R32Acc& acc, const float* tile, const float* mat, int ld, int kp, int np,
                                            int tx, int ty) {
  const float* xr = tile + ty * ld;
  const float* mr = mat + 8 * tx;
#pragma unroll 1
  for (int k = 0; k < kp; k += 4) {
    float4 x[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) x[i] = *reinterpret_cast<const float4*>(xr + 16 * i * ld + k);
#pragma unroll
    for (int kk = 0; kk < 4; ++kk) {
      const ulonglong2 m0 = *reinterpret_cast<const ulonglong2*>(mr + (k + kk) * np);
      const ulonglong2 m1 = *reinterpret_cast<const ulonglong2*>(mr + (k + kk) * np + 4);
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const float v = kk == 0 ? x[i].x : (kk == 1 ? x[i].y : (kk == 2 ? x[i].z : x[i].w));
        const f32x2 vv = pack2(v, v);
        acc[i][0] = fma2(vv, m0.x, acc[i][0]);
        acc[i][1] = fma2(vv, m0.y, acc[i][1]);
        acc[i][2] = fma2(vv, m1.x, acc[i][2]);
        acc[i][3] = fma2(vv, m1.y, acc[i][3]);
      }
    }
  }
}
__device__ __forceinline__ void r32_zero(R32Acc& acc) {
#pragma unroll
  for (int i = 0; i < 8; ++i)
#pragma unroll
    for (int c = 0; c < 4; ++c) acc[i][c] = 0ull;
}
// out rows from the accumulators (sign s), 16 bytes a store where rows allow.
template <class F>
__device__ __forceinline__ void r32_store(const R32Acc& acc, float* g, int rows, int n, int tx, int ty, F add) {
  const bool wide = (n & 3) == 0 && (reinterpret_cast<uintptr_t>(g) & 15) == 0;
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const int r = ty + 16 * i;
    if (r < rows) {
      float v[8];
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        const float2 p = unpack2(acc[i][c]);
        v[2 * c] = add(p.x, r, 8 * tx + 2 * c);
        v[2 * c + 1] = add(p.y, r, 8 * tx + 2 * c + 1);
      }
      float* q = g + static_cast<int64_t>(r) * n + 8 * tx;
      if (wide) {
#pragma unroll
        for (int h = 0; h < 2; ++h)
          if (8 * tx + 4 * h < n)
            *reinterpret_cast<float4*>(q + 4 * h) = make_float4(v[4 * h], v[4 * h + 1], v[4 * h + 2], v[4 * h + 3]);
      } else {
#pragma unroll
        for (int c = 0; c < 8; ++c)
          if (8 * tx + c < n) q[c] = v[c];
      }
    }
  }
}

// Dynamic shared memory: [M1 | M2] matrices, two row tiles.
// out = X M1 + Y M2 (X or Y may be NULL; out may be X or Y: a tile's rows are
// read before they are written).
__global__ void __launch_bounds__(208, 2)
    k_rowmul_f32(const float* X, const double* __restrict__ M1, const float* Y, const double* __restrict__ M2,
                 int64_t m, int n, float* out) {
  extern __shared__ __align__(128) unsigned char smem[];
  const int ld = r32_ld(n), kp = r32_kp(n), np = r32_np(n);
  const int nin = (X ? 1 : 0) + (Y ? 1 : 0);
  float* mat = reinterpret_cast<float*>(smem);
  float* tiles = mat + static_cast<size_t>(nin) * kp * np;
  const int ntx = r32_tx(n), tx = threadIdx.x % ntx, ty = threadIdx.x / ntx;
  for (int i = threadIdx.x; i < nin * kp * np; i += blockDim.x) {
    const int w = i / (kp * np), e = i - w * kp * np, k = e / np, c = e - k * np;
    const double* M = (w == 0 && X) ? M1 : M2;
    mat[i] = k < n && c < n ? static_cast<float>(M[k * n + c]) : 0.0f;
  }
  for (int i = threadIdx.x; i < 2 * kR32Rows * ld; i += blockDim.x) tiles[i] = 0.0f;  // the padding columns
  __syncthreads();
  const int64_t nt = (m + kR32Rows - 1) / kR32Rows;
  auto rows_of = [&](int64_t t) { return static_cast<int>(m - t * kR32Rows < kR32Rows ? m - t * kR32Rows : kR32Rows); };
  int64_t t = blockIdx.x;
  int buf = 0;
  auto load = [&](int64_t tt, int w, int b) {
    if (tt < nt) {
      const float* S = (w == 0 && X) ? X : Y;
      r32_load(tiles + static_cast<size_t>(b) * kR32Rows * ld, S + tt * kR32Rows * n, rows_of(tt), n, ld);
    }
    cp_async_commit();
  };
  load(t, 0, 0);
  for (; t < nt; t += gridDim.x) {
    R32Acc acc;
    r32_zero(acc);
    for (int w = 0; w < nin; ++w) {
      const bool last = w + 1 == nin;
      load(last ? t + gridDim.x : t, last ? 0 : w + 1, buf ^ 1);
      cp_async_wait_1();
      __syncthreads();
      r32_product(acc, tiles + static_cast<size_t>(buf) * kR32Rows * ld, mat + static_cast<size_t>(w) * kp * np, ld, kp,
                  np, tx, ty);
      __syncthreads();  // the tile is free for the copy after the next
      buf ^= 1;
    }
    r32_store(acc, out + t * kR32Rows * n, rows_of(t), n, tx, ty, [](float v, int, int) { return v; });
  }
}

// Step 3 of binary32 data in its own arithmetic (as k_form_q): one CTA per row
// block, tiles last to first, W = T X by the same product.  Yg is overwritten.
__global__ void __launch_bounds__(208, 2)
    k_form_q_f32(float* Yg, int64_t m, int n, int64_t b, int B, int bt, int kt, const double* __restrict__ Tg,
                 const double* __restrict__ Cg, int64_t cblocks) {
  extern __shared__ __align__(128) unsigned char smem[];
  const int ld = r32_ld(n), kp = r32_kp(n), np = r32_np(n);
  float* xm = reinterpret_cast<float*>(smem);
  float* wm = xm + kp * np;
  float* tiles = wm + kp * np;
  const int ntx = r32_tx(n), tx = threadIdx.x % ntx, ty = threadIdx.x / ntx;
  const int64_t row0 = static_cast<int64_t>(blockIdx.x) * b;
  const int64_t rows = m - row0 < b ? m - row0 : b;
  const int ntiles = rows <= B ? 1 : static_cast<int>(1 + (rows - B + bt - 1) / bt);
  const int ntop = static_cast<int>(rows < n ? rows : n);
  const double* Cb = Cg + (cblocks == 1 ? 0 : static_cast<int64_t>(blockIdx.x)) * n * n;
  float* Yb = Yg + row0 * n;
  for (int i = threadIdx.x; i < kp * np; i += blockDim.x) {
    const int k = i / np, c = i - k * np;
    xm[i] = k < n && c < n ? static_cast<float>(Cb[k * n + c]) : 0.0f;
    wm[i] = 0.0f;
  }
  for (int i = threadIdx.x; i < 2 * kR32Rows * ld; i += blockDim.x) tiles[i] = 0.0f;
  __syncthreads();
  for (int t = ntiles - 1; t >= 0; --t) {
    const int64_t tr0 = t == 0 ? 0 : B + static_cast<int64_t>(t - 1) * bt;
    const int cap = t == 0 ? B : bt;
    const int cnt = static_cast<int>(rows - tr0 < cap ? rows - tr0 : cap);
    const bool top = t == 0;
    const double* Tb = Tg + (static_cast<int64_t>(blockIdx.x) * kt + t) * n * n;
    float* tt = tiles;  // T (or Y_top^T) as a tile of n rows
    R32Acc acc;
    const float* src = xm;
    if (top) {  // Z = Y_top^T X, Y_top unit lower triangular
      for (int i = threadIdx.x; i < n * n; i += blockDim.x) {
        const int r = i / n, k = i - r * n;  // row r of Y_top, column k
        tt[k * ld + r] = r < ntop ? (r > k ? Yb[static_cast<int64_t>(r) * n + k] : (r == k ? 1.0f : 0.0f)) : 0.0f;
      }
      __syncthreads();
      r32_zero(acc);
      r32_product(acc, tt, xm, ld, kp, np, tx, ty);
      __syncthreads();
#pragma unroll
      for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int c = 0; c < 4; ++c)
          if (ty + 16 * i < n) *reinterpret_cast<f32x2*>(wm + (ty + 16 * i) * np + 8 * tx + 2 * c) = acc[i][c];
      src = wm;
    }
    for (int i = threadIdx.x; i < n * n; i += blockDim.x) {
      const int r = i / n, k = i - r * n;
      tt[r * ld + k] = k >= r ? f32_of(Tb[i]) : 0.0f;
    }
    __syncthreads();
    r32_zero(acc);
    r32_product(acc, tt, src, ld, kp, np, tx, ty);
    __syncthreads();  // src (xm or wm) and the tile have been read
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        const int o = (ty + 16 * i) * np + 8 * tx + 2 * c;
        if (ty + 16 * i < n) {
          *reinterpret_cast<f32x2*>(wm + o) = acc[i][c];
          if (!top) {  // the coefficient of tile t - 1
            const float2 w = unpack2(acc[i][c]);
            xm[o] -= w.x;
            xm[o + 1] -= w.y;
          }
        }
      }
    // the tile's rows, one piece of 128 ahead
    int buf = 0;
    r32_load(tiles, Yb + tr0 * n, cnt < kR32Rows ? cnt : kR32Rows, n, ld);
    cp_async_commit();
    for (int c0 = 0; c0 < cnt; c0 += kR32Rows, buf ^= 1) {
      const int crows = cnt - c0 < kR32Rows ? cnt - c0 : kR32Rows;
      float* tile = tiles + static_cast<size_t>(buf) * kR32Rows * ld;
      const int nxt = c0 + kR32Rows;
      if (nxt < cnt)
        r32_load(tiles + static_cast<size_t>(buf ^ 1) * kR32Rows * ld, Yb + (tr0 + nxt) * n,
                 cnt - nxt < kR32Rows ? cnt - nxt : kR32Rows, n, ld);
      cp_async_commit();
      cp_async_wait_1();
      __syncthreads();
      if (top && c0 < n) {  // Y_top's upper part is not Y's
        for (int i = threadIdx.x; i < kR32Rows * n; i += blockDim.x) {
          const int r = i / n, k = i - r * n;
          if (k >= c0 + r) tile[r * ld + k] = k == c0 + r && c0 + r < ntop ? 1.0f : 0.0f;
        }
        __syncthreads();
      }
      r32_zero(acc);
      r32_product(acc, tile, wm, ld, kp, np, tx, ty);
      __syncthreads();
      r32_store(acc, Yb + (tr0 + c0) * n, crows, n, tx, ty, [&](float v, int r, int c) {
        return (top && c0 + r < ntop && c < n) ? xm[(c0 + r) * np + c] - v : -v;
      });
    }
    __syncthreads();
  }
}

#endif  // TSQR_ROWS32_KERNELS

}  // namespace tsqr
