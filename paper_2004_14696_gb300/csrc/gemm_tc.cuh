// tcgen05 (5th-generation tensor core) bf16 GEMM for sm_103a, used by the
// worker-gradient pass.  Internal interface.
#pragma once

#include <cuda.h>
#include <cuda_bf16.h>
#include <stdint.h>

#include "common.cuh"

namespace dbw {

enum TcEpiKind { TC_HIDDEN = 0, TC_LOGITS = 1, TC_DX = 2, TC_DW = 3, TC_GBAR = 4 };

// What the epilogue does with accumulator element (m, n) of batch z.
struct TcEpi {
    const float* bias;            // HIDDEN, LOGITS: + bias[n]
    __nv_bfloat16* out;           // HIDDEN, DX: out[m * ldo + n] (bf16, row-major)
    int64_t ldo;
    float* outF;                  // LOGITS: outF[m * ldF + n] (fp32)
    int64_t ldF;
    const __nv_bfloat16* act;     // DX: ReLU mask 1[act[m * ldact + n] > 0]
    int64_t ldact;
    float* G;                     // DW: G[z * ldG + off + m * ldrow + n] (fp32)
    int64_t ldG, off, ldrow;
    // GBAR (mean over the received workers, Eqs. (3)-(4)): with g = acc / k,
    // W[off + m * ldrow + n] -= lr * g, gbar[off + m * ldrow + n] = g (nullable), and the
    // sums of g^2 (fp64) into pieces[(s * ceil(N / 256) + nt) * 8 + h * 4 + q]: rows
    // 128 s + 32 q .. +31 (s < ceil(M / 128)), columns 256 nt + 128 h .. +127.
    float* W;
    float* gbar;
    float lr;
    double* pieces;
    // GBAR, K of the last round's tiles split into ranges when that ends the launch sooner
    // (chosen on the device from the live K; never with part null): the partial sums go to
    // part, tc_split_floats(M, N) floats, and {split tiles, ranges of each, first split tile}
    // to plan[3].  W, gbar and pieces of those tiles are left to the caller.
    float* part;
    int* plan;
    // Live row count on the device: when non-null, only (*kdev) * kmul rows of the
    // row dimension are computed (M for HIDDEN / LOGITS / DX, K for GBAR, where k =
    // *kdev); *kdev <= 0 runs no tile.
    const int* kdev;
    int kmul;
};

// Most K ranges of a GBAR GEMM of M x N over all its split tiles, and their scratch.
int tc_split_items(int M, int N);
size_t tc_split_floats(int M, int N);
constexpr int kTcPartFloats = 32 * 128;   // one block of partial sums

// Operands of one GEMM, both row-major bf16 as their producers left them (ld multiples of
// 8 elements, bases 16-byte aligned):
//   HIDDEN, LOGITS  C[m, n] = sum_k A[m, k] B[n, k]   A [M, lda], B [N, ldb]
//   DX              C[m, n] = sum_k A[m, k] B[k, n]   A [M, lda], B [K, ldb]
//   GBAR            C[m, n] = sum_k A[k, m] B[k, n]   A [K, lda], B [K, ldb]
// An operand whose K runs along its rows is read as an MN-major tile: no transposed copy
// of the weights, the activations or dZ exists.
struct TcOperands {
    const __nv_bfloat16* A;
    int64_t lda;
    const __nv_bfloat16* B;
    int64_t ldb;
    int M, N, K;
};

// The GEMM and then the epilogue ``kind`` (HIDDEN, LOGITS, DX or GBAR).  ``status``
// (device int) gets bit 0 set if a pipeline wait ever times out; it must be zeroed by
// the caller.
int tc_gemm(int kind, const TcOperands& o, const TcEpi& epi, int* status, cudaStream_t st);

// Per-worker weight gradients: for z < batch, C_z[m, n] = sum_{r < B} A[z B + r, m] B_[z B + r, n]
// (A = dZ, o.M = out; o.B = the layer input, o.N = in; o.K = B samples per worker, any
// B >= 1: a worker's rows past B read as zero), stored by the TC_DW epilogue.
int tc_dw(const TcOperands& o, int batch, const TcEpi& epi, int* status, cudaStream_t st);

// 2-D TMA tensor map of a row-major bf16 matrix [rows, cols] with row stride ld
// (elements), box 64 columns (128 bytes, 128-byte swizzle) x box_rows; reads past the
// extents are zero.  False if the driver's encoder is unavailable or rejects the
// arguments.
bool tc_make_map(CUtensorMap* tm, const void* base, int64_t rows, int64_t cols, int64_t ld, int box_rows);

// The same for a row-major fp32 matrix: box 32 (128 bytes, 128-byte swizzle) x box_rows;
// ld a multiple of 4 and base 16-byte aligned.
bool tc_make_map_f32(CUtensorMap* tm, const void* base, int64_t rows, int64_t cols, int64_t ld, int box_rows);
// Row-major fp32 [rows, batch blocks of ld_z columns, the first cols_z of them used]:
// dimensions (column of the block, block, row), box 32 x 1 x box_rows; columns past cols_z
// of a block read as zero.  ld_z a multiple of 4.
bool tc_make_batch_map_f32(CUtensorMap* tm, const void* base, int64_t rows, int64_t batch, int64_t cols_z, int64_t ld_z,
                           int box_rows);

// The mean-gradient GEMM (TC_GBAR, operands g, epilogue ge) and the input-gradient
// GEMM (TC_DX, operands x, epilogue xe) of one layer in one launch: both read dZ_l
// and neither writes what the other reads, so their tiles share the persistent
// grid (those of the mean gradient first).  Same rules as tc_gemm.
int tc_gemm_mean_dx(const TcOperands& g, const TcEpi& ge, const TcOperands& x, const TcEpi& xe, int* status,
                    cudaStream_t st);

// Per-worker squared gradient norms of L layers without forming the gradients, in one
// launch (the Gram identity ||D^T A||_F^2 = <D D^T, A A^T>_F, with the bias term
// ||1^T D||^2 = sum of D D^T added), for each layer l:
//   pieces[l][(r / 32) * CT + ct] = sum over rows r..r+31 of the 32-row group and the
//   columns c of the same worker (in column tile ct, CT = max(1, B / 128)) of
//   (D D^T)[r, c] * ((A A^T)[r, c] + 1)
// for the row groups of the first (*kdev) * B rows.  A = act[l] [rows, ldA[l]] (K =
// colsA[l]), D = dz[l] [rows, ldD] (K = colsD[l]), both bf16 row-major; B % 32 == 0 and
// either 128 % B == 0 or B % 128 == 0.  part: tc_gram_partial_floats(rows, B, L) floats
// of scratch for the partial products of the K ranges; cnt: tc_gram_items(rows, B, L)
// int32 counters, zero on entry and left zero on return.
int tc_gram(int L, const __nv_bfloat16* const* act, const int64_t* ldA, const int* colsA,
            const __nv_bfloat16* const* dz, int64_t ldD, const int* colsD, int rows, int B, const int* kdev,
            double* const* pieces, float* part, int* cnt, int* status, cudaStream_t st);
size_t tc_gram_partial_floats(int rows, int B, int L);
size_t tc_gram_items(int rows, int B, int L);

}  // namespace dbw
