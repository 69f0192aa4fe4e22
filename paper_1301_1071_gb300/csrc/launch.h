// launch.h -- host launchers of the TSQR kernels (internal, C++ linkage).
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

#include "plan.h"

namespace tsqr {

// Lets fn be launched with `bytes` of dynamic shared memory.  The attribute
// belongs to the function, on the whole device: it is set to the same value
// (the most a CTA can have, less a kernel's few static variables) by every call, so
// that a host thread never lowers it between another thread's setting and
// launch.
constexpr size_t kSmemStatic = 128;
template <class F>
inline cudaError_t allow_smem(F* fn, size_t bytes, bool has_static = false) {
  const size_t most = kSmemMax - (has_static ? kSmemStatic : 0);
  if (bytes > most) return cudaErrorInvalidValue;
  return cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(most));
}

// Step 1 / tree level: p CTAs, one per row block of b rows (k.kind selects
// the storage/compute types).
// Blocks of b rows; a block taller than the register tile (b > k.B) is
// factored as tiles of k.B rows and then bt rows, kt tiles at most
// (T slots per block).
cudaError_t launch_local_qr(const KernelCfg& k, const void* A, int64_t m, int n, int64_t b, int64_t bt, int kt,
                            int64_t p, void* Y, double* Rst, double* Tst, int32_t* status, cudaStream_t st);
// Step 1 of binary64 data by panels (tiles of kPdRows rows, kt T slots per block):
// Y, R and tau, or (Y == NULL) R only.
cudaError_t launch_panel_qr_f64(const PanelCfg& k, const void* A, int64_t m, int n, int64_t b, int kt, int64_t p,
                                void* Y, double* Rst, double* Tst, int32_t* status, cudaStream_t st);
// Step 3: p CTAs (B, bt: the tile geometry of Step 1; comp: the T slots hold 2 -
// tau, comp_at; rows32: Plan's).
cudaError_t launch_form_q(const KernelCfg& k, const void* Y, int64_t m, int n, int64_t b, int B, int64_t bt, int kt,
                          int64_t p, const double* T, const double* C, int64_t cblocks, bool comp, bool rows32,
                          void* Q, int32_t* status, cudaStream_t st);

// Step-2 up pass of one tree level (binary64): node b = f stacked
// triangular blocks of X (rows x n) -> its R (raw signs) into Rout's block
// b; with Y (may alias X): the Householder vectors over the node's rows and
// tau + Gram entries into the node's T slot (Tst); Y == NULL: R only.
// tree_up_fits: the node fits one CTA's shared memory.  tree_up_cl_fits:
// the node fits a cluster of f CTAs, one block each (launch_tree_up_cl, same
// outputs).  Neither: the row-block kernel takes the level.
constexpr int kTreeClMaxF = 8;  // portable cluster size
constexpr int kTreeCompMinN = 3;  // comp_at's least n
bool tree_up_fits(int n, int f);
cudaError_t launch_tree_up(const double* X, int64_t rows, int n, int f, int64_t p, double* Y, double* Rout,
                           double* Tst, cudaStream_t st);
bool tree_up_cl_fits(int n, int f);
cudaError_t launch_tree_up_cl(const double* X, int64_t rows, int n, int f, int64_t p, double* Y, double* Rout,
                              double* Tst, cudaStream_t st);

// Step-2 down pass of one tree level (binary64): node b's rows of Y (f
// stacked blocks of n rows, the last node possibly fewer) become its
// children's coefficient blocks from C (cblocks == 1: one block for all),
// using Y = [I; V_2; ...; V_f] with V_k upper triangular.  comp: the T slots
// hold 1 - tau (launch_tree_up's, n >= kTreeCompMinN).
cudaError_t launch_tree_down(double* Y, int64_t rows, int n, int f, int64_t p, const double* T, const double* C,
                             int64_t cblocks, bool comp, cudaStream_t st);

// Step 3 for binary32 data on the tensor cores (3xTF32), n <= 100; the block
// and tile geometry (b, B = the Step-1 register tile, bt, kt) of Step 1.  For
// n <= 64 the T slots and C are overwritten (with W and X_0).
cudaError_t launch_form_q_tc(float* Y, int64_t m, int n, int64_t b, int B, int64_t bt, int kt, int64_t p,
                             double* T, double* C, int64_t cblocks, int32_t* status, cudaStream_t st);

// out_r = X_r M1 + Y_r M2 over p blocks of b rows (X or Y may be NULL).
cudaError_t launch_rowmul(const KernelCfg& k, const void* X, const double* M1, const void* Y,
                          const double* M2, int64_t m, int n, int64_t b, int64_t p, void* out, int32_t* status,
                          cudaStream_t st);
// Partial Grams X^T Y (grid partials of n x n binary64), then their fixed-order sum into G.
// acc_storage: per-CTA partial Grams accumulate in the storage type (binary32
// data: the FMA pipe); the cross-CTA sum is always binary64.  binary64 data:
// launch_gram_split (colexp passed to it).  max_parts: the partials that part holds.
cudaError_t launch_gram(int esz, const void* X, const void* Y, int64_t m, int n, double* part, double* G,
                        int max_parts, int32_t* status, cudaStream_t st, bool acc_storage = false,
                        int* colexp = nullptr);

// binary64 as exact digit products (split_kernels.cuh).  out (+)= X M, n <=
// kRsMaxN: colsrc / colexp give the scale of X's columns (see k_rowmul_split).
// kSplitMinN: below, the padding to 8 columns and 16 k steps costs more than
// the binary64 unit (GB300, 20,000,000 x 4: Cholesky QR 2.6 ms by FMAs, 5.4 by
// digits, direct 2.9 against 4.1; 10,000,000 x 6 direct 3.91 against 3.91; at
// 10,000,000 x 8 5.1 against 4.6).
constexpr int kSplitMinN = 7;
constexpr int kRowSplitMaxN = 64;
constexpr bool rows_by_digits(int64_t n) { return n >= kSplitMinN && n <= kRowSplitMaxN; }
cudaError_t launch_rowmul_split(const double* X, const double* M, const double* colsrc, const int* colexp, int64_t m,
                                int n, bool add, double* out, int32_t* status, cudaStream_t st);
// Step 3 for binary64 data, n <= kRowSplitMaxN; the block and tile geometry of
// Step 1, Q over Y.  comp: the T slots hold 2 - tau (comp_at).
cudaError_t launch_form_q_split(double* Y, int64_t m, int n, int64_t b, int B, int64_t bt, int kt, int64_t p,
                                const double* T, const double* C, int64_t cblocks, bool comp, int32_t* status,
                                cudaStream_t st);
// Partial Grams X^T Y into at most max_parts n x n partials (*parts written);
// colexp (or NULL): n ints, zeroed by the caller, receiving the largest binary
// exponents of X's columns.
cudaError_t launch_gram_split(const double* X, const double* Y, int64_t m, int n, int max_parts, int* parts,
                              double* part, int* colexp, cudaStream_t st);
// X^T X of binary32 data with binary64 accuracy (Cholesky QR), n >=
// kGramSplitF32MinN: below, binary64 FMAs take no longer (Cholesky QR of
// 3,000,000 x 9: 1.73 ms by FMAs, 2.15 by digits; x 12: 2.71 and 1.49).
constexpr int kGramSplitF32MinN = 12;
cudaError_t launch_gram_split_f32(const float* X, int64_t m, int n, int max_parts, int* parts, double* part,
                                  cudaStream_t st);
// The Gram entries of every tile's Householder vectors into the T slots'
// strictly upper triangles.
cudaError_t launch_gram_t_split(const double* Y, int64_t m, int n, int64_t b, int B, int64_t bt, int kt, int64_t p,
                                double* T, cudaStream_t st);

// binary32 row products in 128-row tiles (rows32.cuh): out = X M1 + Y M2 (either
// input NULL; out may be an input), and Step 3 in binary32 arithmetic (Q over Y).
// Rows times a matrix, GB300, the earlier kernel / this: n = 8 at 300,000 rows 1.43,
// n = 13 .. 61 odd 0.93 to 1.25, n = 64 1.39 to 1.65; but rows of odd length are
// copied 4 bytes at a time, and above n = 64 one CTA an SM is left: 1,500,000 x 69
// 0.78, 77 0.85, 81 0.99, 89 1.08: odd n from 65 to 80 keep k_rowmul.
constexpr int kRows32MinN = 8;
constexpr bool rowmul_rows32(int64_t n) { return n >= kRows32MinN && (n <= 64 || n > 80 || n % 2 == 0); }
// Step 3 of p row blocks: a CTA has 16 ceil(n / 8) threads here, 128 and more in
// k_form_q, so narrow matrices need several CTAs an SM to gain.  k_form_q's time
// over this, blocks of 1,024 rows or the planner's: n = 52 .. 64 1.03 to 3.9 at any
// p; n = 33 .. 50 0.66 to 0.97 at 1 .. 147 blocks, 1.12 to 2.2 from 293 on; n = 16 ..
// 29 0.5 to 1.0 up to 293 blocks, 0.94 to 2.06 at 586 and more; n = 8 .. 15 0.5 to
// 1.0 at 608 (tall ones too), from 1,465 on 1.1 to 1.9 but for 13 and 15 (0.91,
// 0.94).  Odd n > 64 as above (2,000,000 x 77 with adjoint 16.5 ms in k_form_q, 16.8
// here), even ones 1.02 to 1.6 at any p.
constexpr bool step3_rows32(int n, int64_t p, int64_t sms) {
  return n < kRows32MinN || (n > 64 && n % 2) ? false
         : n >= 52                            ? true
         : n >= 32                            ? 4 * p >= 7 * sms
         : n >= 16                            ? p >= 3 * sms
                                              : p >= 8 * sms && !(n >= 13 && n % 2);
}
cudaError_t launch_rowmul_f32_tiles(const float* X, const double* M1, const float* Y, const double* M2, int64_t m,
                                    int n, float* out, cudaStream_t st);
cudaError_t launch_form_q_f32_tiles(float* Y, int64_t m, int n, int64_t b, int B, int64_t bt, int kt, int64_t p,
                                    const double* T, const double* C, int64_t cblocks, cudaStream_t st);

// Gram launch geometry shared by the planner and the launcher.
struct GramGeom { int chunk, grid, nt, tile; };
GramGeom gram_geom(int64_t m, int n, int esz, bool small = false);

}  // namespace tsqr
