// Eq. (2) for all n workers at once (fp32, and bf16 where grads_tc.cu does not take it): g_i = (1/B) sum_{x in B_i} grad f(x, w).
//
// The n workers share w, so their minibatches are stacked into one batch of
// M = n * B rows and every forward and input-gradient GEMM is a single GEMM over
// M rows.  Only the weight gradient is per worker: G[i, W_l] = dZ_l[i]^T A_{l-1}[i]
// with K = B, a batched GEMM over the n workers that writes G directly.
//
//   gather     X = pool[idx] in the operand type (fp32: a single layer of at most 16 outputs
//              reads the pool itself)
//   forward    Z_l = A_{l-1} W_l^T + b_l, A_l = ReLU(Z_l)   (last layer: fp32 logits)
//   loss       per-sample cross entropy, loss_i = mean over worker i's B samples,
//              dZ_L = (softmax - onehot) / B (fp32, at most 16 outputs: one launch with the
//              last layer's forward)
//   backward   G[i, W_l] = dZ_l[i]^T A_{l-1}[i],  G[i, b_l] = sum_rows dZ_l[i],
//              dZ_{l-1} = (dZ_l W_l) * 1[A_{l-1} > 0]      (ReLU'(0) = 0)
//
// The large forward and weight-gradient GEMMs run on the tensor cores in three tf32
// passes (gemm_tf32.cuh), which keeps fp32 accuracy; the others are FFMA kernels on fp32 or
// bf16 operands.
#include <math.h>

#include <type_traits>

#include "common.cuh"
#include "gemm_tf32.cuh"
#include "grads.cuh"
#include "loss_bias.cuh"
#include "tc_ptx.cuh"

namespace dbw {

namespace tf32 {
__global__ void split_kernel(const float* __restrict__ src, int rows, int cols, int64_t lds, float* __restrict__ hi,
                             float* __restrict__ lo, int64_t ldo) {
    grid_begin();
    for (int r = blockIdx.y; r < rows; r += gridDim.y) {
        const float* s = src + (int64_t)r * lds;
        for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < cols; c += gridDim.x * blockDim.x) {
            float h, l;
            split_value(s[c], h, l);
            hi[(int64_t)r * ldo + c] = h;
            lo[(int64_t)r * ldo + c] = l;
        }
    }
}

__global__ void split4_kernel(const float* __restrict__ src, int rows, int cols, int64_t lds, float* __restrict__ hi,
                              float* __restrict__ lo, int64_t ldo) {
    grid_begin();
    const int c4 = cols / 4;
    const int64_t total = (int64_t)rows * c4;
    for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < total; q += (int64_t)gridDim.x * blockDim.x) {
        const int64_t r = q / c4;
        const int c = static_cast<int>(q - r * c4) * 4;
        const float4 v = *reinterpret_cast<const float4*>(src + r * lds + c);
        float4 h, l;
        split_value(v.x, h.x, l.x);
        split_value(v.y, h.y, l.y);
        split_value(v.z, h.z, l.z);
        split_value(v.w, h.w, l.w);
        *reinterpret_cast<float4*>(hi + r * ldo + c) = h;
        *reinterpret_cast<float4*>(lo + r * ldo + c) = l;
    }
}

void split(const float* src, int rows, int cols, int64_t lds, float* hi, float* lo, int64_t ldo, cudaStream_t st) {
    if (cols % 4 == 0 && lds % 4 == 0 && ldo % 4 == 0 && aligned16(src) && aligned16(hi) && aligned16(lo)) {
        const int64_t want = ((int64_t)rows * (cols / 4) + 255) / 256;
        const int blocks = static_cast<int>(want < 8 * sm_count() ? want : 8 * sm_count());
        launch(split4_kernel, blocks < 1 ? 1 : blocks, 256, 0, st, src, rows, cols, lds, hi, lo, ldo);
    } else {
        dim3 g((cols + 127) / 128, rows < 65535 ? rows : 65535);
        launch(split_kernel, g, 128, 0, st, src, rows, cols, lds, hi, lo, ldo);
    }
}

__global__ void split_t_kernel(const float* __restrict__ src, int rows, int cols, int64_t lds, int B, int pad,
                               float* __restrict__ hiT, float* __restrict__ loT, int64_t ldt) {
    grid_begin();
    __shared__ float tile[32][33];
    const int tx = threadIdx.x, ty = threadIdx.y;
    const int c0 = blockIdx.x * 32;
    for (int64_t r0 = (int64_t)blockIdx.y * 32; r0 < rows; r0 += (int64_t)gridDim.y * 32) {
        for (int j = ty; j < 32; j += 8) {
            const int64_t r = r0 + j;
            const int c = c0 + tx;
            tile[j][tx] = (r < rows && c < cols) ? src[r * lds + c] : 0.f;
        }
        __syncthreads();
        const int64_t r = r0 + tx;
        const int64_t t = pad ? r + static_cast<int>(r) / B * pad : r;
        for (int j = ty; j < 32; j += 8) {
            const int c = c0 + j;
            if (c < cols && r < rows) {
                float h, l;
                split_value(tile[tx][j], h, l);
                hiT[(int64_t)c * ldt + t] = h;
                loT[(int64_t)c * ldt + t] = l;
            }
        }
        __syncthreads();
    }
}
}  // namespace tf32

namespace {

// ------------------------------------------------------------------ gather
__device__ __forceinline__ float to_f(float v) { return v; }
__device__ __forceinline__ float to_f(__nv_bfloat16 v) { return __bfloat162float(v); }

// X[m, :] = pool[idx[m], :] in the operand type, 16 bytes a lane (in % 4 == 0).  An index
// outside [0, S) reads row 0; the loss kernel poisons that worker.
template <typename T>
__global__ void gather_kernel(const float* __restrict__ pool, int64_t S, int in, const int32_t* __restrict__ idx,
                              int M, T* __restrict__ X) {
    grid_begin();
    for (int m = blockIdx.y; m < M; m += gridDim.y) {
        int64_t r = idx[m];
        if (r < 0 || r >= S) r = 0;
        const float4* src = reinterpret_cast<const float4*>(pool + r * in);
        T* dst = X + (int64_t)m * in;
        for (int c = blockIdx.x * blockDim.x + threadIdx.x; 4 * c < in; c += gridDim.x * blockDim.x) {
            const float4 v = src[c];
            if constexpr (sizeof(T) == 4)
                reinterpret_cast<float4*>(dst)[c] = v;
            else   // rows of in bf16 start on 8 bytes
                reinterpret_cast<uint2*>(dst)[c] = make_uint2(tcx::pack_bf16(v.x, v.y), tcx::pack_bf16(v.z, v.w));
        }
    }
}

// bf16 copy of the weights (the flat layout of w; the bias slots are not read).
__global__ void cast_bf16_kernel(const float* __restrict__ w, int64_t d, __nv_bfloat16* __restrict__ wb) {
    grid_begin();
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < d; i += (int64_t)gridDim.x * blockDim.x)
        wb[i] = __float2bfloat16_rn(w[i]);
}

// The gather of the fp32 pass when its first layer runs in three tf32 passes: the
// gathered rows' tf32 parts row-major (hi / lo [M, ldo], when hi != nullptr) and
// transposed (hiT / loT [in, ldt], when hiT != nullptr: the workers' B samples in blocks of
// B + pad columns), and X itself when X != nullptr.
// Tiles of 32 rows x 128 columns through shared memory, blocks of 32 x 8 threads: a lane
// moves 16 bytes of a row (in, ldo multiples of 4), then 4-byte pieces of the transposed
// rows, 128 contiguous bytes a warp.  The blocks from row ``ty_n`` of the grid on split the first
// layer's weights (W, nw4 groups of 4, into w_hi / w_lo), and the first block zeroes the status
// word and the loss counters (zero[0 .. nzero)): three launches in one (784-256-10: 64 workers of 64
// samples 120.1 -> 116.3 us an iteration, gradients of 16 of 500 174.5 -> 168.8).
__global__ void gather_parts_kernel(int ty_n, const float* __restrict__ W, int64_t nw4, float* __restrict__ w_hi,
                                    float* __restrict__ w_lo, int* __restrict__ zero, int nzero,
                                    const float* __restrict__ pool, int64_t S, int in,
                                    const int32_t* __restrict__ idx, int M, float* __restrict__ X,
                                    float* __restrict__ hi, float* __restrict__ lo, int64_t ldo,
                                    float* __restrict__ hiT, float* __restrict__ loT, int64_t ldt, int B, int pad) {
    grid_begin();
    __shared__ float tile[32][129];   // [row][column], padded: the transposed reads are conflict-free
    const int tx = threadIdx.x, ty = threadIdx.y;
    if (static_cast<int>(blockIdx.y) >= ty_n) {
        const int64_t first = ((int64_t)(blockIdx.y - ty_n) * gridDim.x + blockIdx.x) * 256 + ty * 32 + tx;
        const int64_t step = (int64_t)(gridDim.y - ty_n) * gridDim.x * 256;
        for (int64_t e = first; e < nw4; e += step) {
            const float4 v = reinterpret_cast<const float4*>(W)[e];
            float4 h, l;
            tf32::split_value(v.x, h.x, l.x);
            tf32::split_value(v.y, h.y, l.y);
            tf32::split_value(v.z, h.z, l.z);
            tf32::split_value(v.w, h.w, l.w);
            reinterpret_cast<float4*>(w_hi)[e] = h;
            reinterpret_cast<float4*>(w_lo)[e] = l;
        }
        return;
    }
    if (blockIdx.x == 0 && blockIdx.y == 0)
        for (int e = ty * 32 + tx; e < nzero; e += 256) zero[e] = 0;
    const int c0 = blockIdx.x * 128;
    for (int64_t m0 = (int64_t)blockIdx.y * 32; m0 < M; m0 += (int64_t)ty_n * 32) {
        // the four rows' indices, then their four loads in flight together
        const int c = c0 + 4 * tx;
        int64_t src[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int64_t m = m0 + ty + 8 * u;
            src[u] = m < M ? idx[m] : 0;
            if (src[u] < 0 || src[u] >= S) src[u] = 0;
        }
        float4 x[4];
#pragma unroll
        for (int u = 0; u < 4; ++u)
            x[u] = m0 + ty + 8 * u < M && c < in ? *reinterpret_cast<const float4*>(pool + src[u] * in + c)
                                                 : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int j = ty + 8 * u;
            const int64_t m = m0 + j;
            const float4 v = x[u];
            if (m < M && c < in) {
                if (X) *reinterpret_cast<float4*>(X + m * in + c) = v;
                if (hi) {
                    float4 h, l;
                    tf32::split_value(v.x, h.x, l.x);
                    tf32::split_value(v.y, h.y, l.y);
                    tf32::split_value(v.z, h.z, l.z);
                    tf32::split_value(v.w, h.w, l.w);
                    *reinterpret_cast<float4*>(hi + m * ldo + c) = h;
                    *reinterpret_cast<float4*>(lo + m * ldo + c) = l;
                }
            }
            tile[j][4 * tx] = v.x;
            tile[j][4 * tx + 1] = v.y;
            tile[j][4 * tx + 2] = v.z;
            tile[j][4 * tx + 3] = v.w;
        }
        if (hiT) {
            __syncthreads();
            const int64_t m = m0 + tx;
            const int64_t t = pad ? m + static_cast<int>(m) / B * pad : m;
            for (int cc = ty; cc < 128; cc += 8) {
                const int c = c0 + cc;
                if (c < in && m < M)
                    tf32::split_value(tile[tx][cc], hiT[(int64_t)c * ldt + t], loT[(int64_t)c * ldt + t]);
            }
            __syncthreads();
        }
    }
}

// ------------------------------------------------------------------ SIMT GEMM
// C[m, n] = sum_k A(m, k) B(k, n) over a 128 x 128 tile per CTA, 16-deep K
// slices staged in shared memory as fp32, 8 x 8 outputs per thread.  Two shared
// buffers: the next slice's global loads go to registers while the current slice
// is multiplied, then to the other buffer (every output still adds its products
// in increasing k).
//   A_K: A(m,k) = A[m*lda + k]   else A(m,k) = A[k*lda + m]
//   B_K: B(k,n) = B[n*ldb + k]   else B(k,n) = B[k*ldb + n]
// blockIdx.z is a batch index (offsets batchA / batchB).
constexpr int BM = 128, BN = 128, BK = 16;

// SPLIT (unbatched GEMMs with few output tiles): blockIdx.z is a split of K
// instead of a batch index; split z covers k in [z * kps, (z + 1) * kps) and
// writes its partial tile to part[z][M][N], which splitk_reduce_kernel sums in
// split order before the epilogue.
template <typename T, bool A_K, bool B_K, class Epi, bool SPLIT>
__global__ void __launch_bounds__(256) gemm_simt_kernel(int M, int N, int K, const T* __restrict__ A, int64_t lda,
                                                        int64_t batchA, const T* __restrict__ B, int64_t ldb,
                                                        int64_t batchB, Epi epi, int kps, float* __restrict__ part) {
    grid_begin();
    __shared__ __align__(16) float As[2][BK][BM];
    __shared__ __align__(16) float Bs[2][BK][BN];
    const int z = blockIdx.z;
    if (!SPLIT) {
        A += (int64_t)z * batchA;
        B += (int64_t)z * batchB;
    }
    const int kbeg = SPLIT ? z * kps : 0;
    const int kend = SPLIT ? (kbeg + kps < K ? kbeg + kps : K) : K;
    const int m0 = blockIdx.y * BM, n0 = blockIdx.x * BN;
    const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
    float acc[8][8];
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int j = 0; j < 8; ++j) acc[i][j] = 0.f;

    constexpr int LA = BM * BK / 256, LB = BN * BK / 256;   // elements per thread and slice
    float ra[LA], rb[LB];
    // global -> registers: the slice starting at k0 (element e of the tile is thread e % 256's)
    auto load = [&](int k0) {
#pragma unroll
        for (int q = 0; q < LA; ++q) {
            const int e = tid + q * 256;
            int mm, kk;
            if (A_K) { mm = e / BK; kk = e % BK; } else { kk = e / BM; mm = e % BM; }
            const int gm = m0 + mm, gk = k0 + kk;
            ra[q] = (gm < M && gk < kend) ? to_f(A_K ? A[(int64_t)gm * lda + gk] : A[(int64_t)gk * lda + gm]) : 0.f;
        }
#pragma unroll
        for (int q = 0; q < LB; ++q) {
            const int e = tid + q * 256;
            int nn, kk;
            if (B_K) { nn = e / BK; kk = e % BK; } else { kk = e / BN; nn = e % BN; }
            const int gn = n0 + nn, gk = k0 + kk;
            rb[q] = (gn < N && gk < kend) ? to_f(B_K ? B[(int64_t)gn * ldb + gk] : B[(int64_t)gk * ldb + gn]) : 0.f;
        }
    };
    // registers -> shared buffer ``buf``
    auto store = [&](int buf) {
#pragma unroll
        for (int q = 0; q < LA; ++q) {
            const int e = tid + q * 256;
            if (A_K) As[buf][e % BK][e / BK] = ra[q]; else As[buf][e / BM][e % BM] = ra[q];
        }
#pragma unroll
        for (int q = 0; q < LB; ++q) {
            const int e = tid + q * 256;
            if (B_K) Bs[buf][e % BK][e / BK] = rb[q]; else Bs[buf][e / BN][e % BN] = rb[q];
        }
    };
    if (kbeg < kend) {
        load(kbeg);
        store(0);
    }
    __syncthreads();
    int buf = 0;
    for (int k0 = kbeg; k0 < kend; k0 += BK) {
        const bool more = k0 + BK < kend;
        if (more) load(k0 + BK);   // in flight while this slice is multiplied
#pragma unroll
        for (int kk = 0; kk < BK; ++kk) {
            const float4 a0 = *reinterpret_cast<const float4*>(&As[buf][kk][ty * 4]);
            const float4 a1 = *reinterpret_cast<const float4*>(&As[buf][kk][64 + ty * 4]);
            const float4 b0 = *reinterpret_cast<const float4*>(&Bs[buf][kk][tx * 4]);
            const float4 b1 = *reinterpret_cast<const float4*>(&Bs[buf][kk][64 + tx * 4]);
            const float a[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
            const float b[8] = {b0.x, b0.y, b0.z, b0.w, b1.x, b1.y, b1.z, b1.w};
#pragma unroll
            for (int i = 0; i < 8; ++i)
#pragma unroll
                for (int j = 0; j < 8; ++j) acc[i][j] = fmaf(a[i], b[j], acc[i][j]);
        }
        // the other buffer was last read before the previous barrier
        if (more) store(buf ^ 1);
        __syncthreads();
        buf ^= 1;
    }
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const int gm = m0 + (i < 4 ? ty * 4 + i : 64 + ty * 4 + (i - 4));
        if (gm >= M) continue;
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const int gn = n0 + (j < 4 ? tx * 4 + j : 64 + tx * 4 + (j - 4));
            if (gn < N) {
                if (SPLIT)
                    part[((int64_t)z * M + gm) * N + gn] = acc[i][j];
                else
                    epi(z, gm, gn, acc[i][j]);
            }
        }
    }
}

// Sum of the splits of every output element, in split order, then the epilogue.
template <class Epi>
__global__ void splitk_reduce_kernel(int M, int N, int splits, const float* __restrict__ part, Epi epi) {
    grid_begin();
    const int64_t total = (int64_t)M * N;
    for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < total; q += (int64_t)gridDim.x * blockDim.x) {
        float v = 0.f;
        for (int sp = 0; sp < splits; ++sp) v += part[sp * total + q];
        epi(0, static_cast<int>(q / N), static_cast<int>(q % N), v);
    }
}

// forward hidden layer: A_l = ReLU(C + b)
template <typename T>
struct EpiHidden {
    const float* bias;
    T* out;
    int ldo;
    __device__ __forceinline__ void operator()(int, int m, int n, float v) const {
        v += bias[n];
        out[(int64_t)m * ldo + n] = from_f<T>(v > 0.f ? v : 0.f);
    }
    // 32 consecutive outputs of row m from column n0 (those below N): the biases are
    // loaded before any store
    __device__ __forceinline__ void row32(int m, int n0, int N, const float (&v)[32]) const {
        float b[32];
#pragma unroll
        for (int j = 0; j < 32; ++j) b[j] = n0 + j < N ? bias[n0 + j] : 0.f;
#pragma unroll
        for (int j = 0; j < 32; ++j) {
            const float x = v[j] + b[j];
            if (n0 + j < N) out[(int64_t)m * ldo + n0 + j] = from_f<T>(x > 0.f ? x : 0.f);
        }
    }
};
// forward last layer: logits = C + b (fp32)
struct EpiLogits {
    const float* bias;
    float* out;
    int ldo;
    __device__ __forceinline__ void operator()(int, int m, int n, float v) const {
        out[(int64_t)m * ldo + n] = v + bias[n];
    }
    __device__ __forceinline__ void row32(int m, int n0, int N, const float (&v)[32]) const {
        float b[32];
#pragma unroll
        for (int j = 0; j < 32; ++j) b[j] = n0 + j < N ? bias[n0 + j] : 0.f;
#pragma unroll
        for (int j = 0; j < 32; ++j)
            if (n0 + j < N) out[(int64_t)m * ldo + n0 + j] = v[j] + b[j];
    }
};
// input gradient: dZ_{l-1} = C * 1[A_{l-1} > 0]  (a product, so a NaN-poisoned row stays NaN)
template <typename T>
struct EpiDx {
    const T* act;
    T* out;
    int ldo;
    __device__ __forceinline__ void operator()(int, int m, int n, float v) const {
        const float a = to_f(act[(int64_t)m * ldo + n]);
        out[(int64_t)m * ldo + n] = from_f<T>(v * (a > 0.f ? 1.f : 0.f));
    }
};
// weight gradient of worker z: G[z, off + o * in + c]
struct EpiDW {
    float* G;
    int64_t ldG;
    int64_t off;
    int in;
    __device__ __forceinline__ void operator()(int z, int o, int c, float v) const {
        G[(int64_t)z * ldG + off + (int64_t)o * in + c] = v;
    }
};

// Splits of K for an unbatched GEMM with few output tiles: enough CTAs for about
// two per SM, each split at least 4 K blocks deep; 1 = no split.
int splitk_count(int M, int N, int K, int batch) {
    if (batch != 1) return 1;
    const int tiles = ((N + BN - 1) / BN) * ((M + BM - 1) / BM);
    const int want = (2 * sm_count() + tiles - 1) / tiles;
    const int most = K / (4 * BK);
    int s = want < most ? want : most;
    return s < 1 ? 1 : s;
}

// Fills dst[e] = f(e) for e < count, each thread loading 8 values before storing any
// (so that one thread's loads are in flight together, not one per store).
template <class F>
__device__ __forceinline__ void fill_shared(float* dst, int count, F f) {
    for (int e0 = threadIdx.x; e0 < count; e0 += 8 * blockDim.x) {
        float t[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const int e = e0 + u * blockDim.x;
            t[u] = e < count ? f(e) : 0.f;
        }
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const int e = e0 + u * blockDim.x;
            if (e < count) dst[e] = t[u];
        }
    }
}

// ------------------------------------------------------------------ skinny GEMMs
// Forward GEMM with few outputs (the logits): C[m, n] = sum_k A[m, k] W[n, k] for
// N <= kSkinnyN.  W sits in shared memory; one warp per row of A, lane l taking
// k = l, l + 32, .. (coalesced) into N partial sums, which a butterfly adds across the
// warp; lane n hands output n to the epilogue.
constexpr int kSkinnyN = 16;
constexpr int kSkinnyK = 32;
constexpr size_t kSkinnySmem = 48 * 1024;

template <typename T, class Epi>
__global__ void __launch_bounds__(256) skinny_n_kernel(int M, int N, int K, const T* __restrict__ A, int64_t lda,
                                                       const T* __restrict__ W, int64_t ldw, Epi epi) {
    grid_begin();
    extern __shared__ float wsh[];   // W as [N, K] fp32
    fill_shared(wsh, N * K, [&](int e) { return to_f(W[(int64_t)(e / K) * ldw + e % K]); });
    __syncthreads();
    const int lane = threadIdx.x & 31;
    const int nwarps = (gridDim.x * blockDim.x) >> 5;
    for (int m = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; m < M; m += nwarps) {
        float acc[kSkinnyN];
#pragma unroll
        for (int n = 0; n < kSkinnyN; ++n) acc[n] = 0.f;
        const T* a = A + (int64_t)m * lda;
        // 8 of the lane's elements loaded at a time, then multiplied
        for (int k0 = lane; k0 < K; k0 += 8 * 32) {
            float av[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) av[u] = k0 + 32 * u < K ? to_f(a[k0 + 32 * u]) : 0.f;
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const int k = k0 + 32 * u;
                if (k < K) {
#pragma unroll
                    for (int n = 0; n < kSkinnyN; ++n)
                        if (n < N) acc[n] = fmaf(av[u], wsh[n * K + k], acc[n]);
                }
            }
        }
        float mine = 0.f;
#pragma unroll
        for (int n = 0; n < kSkinnyN; ++n) {
            if (n < N) {
                float v = acc[n];
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
                if (lane == n) mine = v;
            }
        }
        if (lane < N) epi(0, m, lane, mine);
    }
}

// The same for fp32 operands whose rows allow 16-byte loads (K, lda, ldw multiples of 4,
// A and W 16-byte aligned): no shared memory, W read through L1; lane l takes the
// 4-element groups k = 4 l, 4 l + 128, .. of its row, each group's products added in k
// order, then the butterfly.
// kTwo: two groups per pass with all their loads issued first (fewer round trips for long
// rows, at about 160 registers); else one group per pass (few registers, for K <= 256).
template <bool kTwo>
__device__ __forceinline__ float skinny_row(const float* __restrict__ a, const float* __restrict__ W, int64_t ldw, int N,
                                            int K, int lane) {
    float acc[kSkinnyN];
#pragma unroll
    for (int n = 0; n < kSkinnyN; ++n) acc[n] = 0.f;
    if constexpr (kTwo) {
        // two of the lane's 4-element groups per pass, all their loads issued before the
        // products (which are added in group order, as below)
        for (int k0 = 4 * lane; k0 < K; k0 += 256) {
            const bool two = k0 + 128 < K;
            const float4 av0 = __ldg(reinterpret_cast<const float4*>(a + k0));
            const float4 av1 =
                two ? __ldg(reinterpret_cast<const float4*>(a + k0 + 128)) : make_float4(0.f, 0.f, 0.f, 0.f);
            float4 wv0[kSkinnyN], wv1[kSkinnyN];
#pragma unroll
            for (int n = 0; n < kSkinnyN; ++n) {
                if (n < N) {
                    wv0[n] = __ldg(reinterpret_cast<const float4*>(W + (int64_t)n * ldw + k0));
                    if (two) wv1[n] = __ldg(reinterpret_cast<const float4*>(W + (int64_t)n * ldw + k0 + 128));
                }
            }
#pragma unroll
            for (int n = 0; n < kSkinnyN; ++n) {
                if (n < N) {
                    float t = acc[n];
                    t = fmaf(av0.x, wv0[n].x, t);
                    t = fmaf(av0.y, wv0[n].y, t);
                    t = fmaf(av0.z, wv0[n].z, t);
                    t = fmaf(av0.w, wv0[n].w, t);
                    if (two) {
                        t = fmaf(av1.x, wv1[n].x, t);
                        t = fmaf(av1.y, wv1[n].y, t);
                        t = fmaf(av1.z, wv1[n].z, t);
                        t = fmaf(av1.w, wv1[n].w, t);
                    }
                    acc[n] = t;
                }
            }
        }
    } else {
        for (int k = 4 * lane; k < K; k += 128) {
            const float4 av = __ldg(reinterpret_cast<const float4*>(a + k));
#pragma unroll
            for (int n = 0; n < kSkinnyN; ++n) {
                if (n < N) {
                    const float4 wv = __ldg(reinterpret_cast<const float4*>(W + (int64_t)n * ldw + k));
                    float t = acc[n];
                    t = fmaf(av.x, wv.x, t);
                    t = fmaf(av.y, wv.y, t);
                    t = fmaf(av.z, wv.z, t);
                    t = fmaf(av.w, wv.w, t);
                    acc[n] = t;
                }
            }
        }
    }
    float mine = 0.f;
#pragma unroll
    for (int n = 0; n < kSkinnyN; ++n) {
        if (n < N) {
            float v = acc[n];
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
            if (lane == n) mine = v;
        }
    }
    return mine;
}

template <bool kTwo, class Epi>
__global__ void __launch_bounds__(128) skinny_n4_kernel(int M, int N, int K, const float* __restrict__ A, int64_t lda,
                                                        const float* __restrict__ W, int64_t ldw, Epi epi) {
    grid_begin();
    const int lane = threadIdx.x & 31;
    const int nwarps = (gridDim.x * blockDim.x) >> 5;
    for (int m = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; m < M; m += nwarps) {
        const float mine = skinny_row<kTwo>(A + (int64_t)m * lda, W, ldw, N, K, lane);
        if (lane < N) epi(0, m, lane, mine);
    }
}

// The last layer with few outputs and the loss in one launch: a warp forms its row's logits as
// above and, lane c holding class c, the sample loss and the row of dZ_L as the loss kernel
// does (the same exchanges, so the same bits).  CTA (x, i) takes rows x rows_cta .. of worker i.
// Of a one-layer model the rows come straight from the pool (``pool`` non-null; an index
// outside [0, S) reads row 0).  These passes are chains of launches of a few us each: with the
// logits and the loss apart, and a gather before a single layer, 784-10 at 16 workers of 32
// took 32.3 us an iteration in a graph, 784-256-10 at 64 of 64 125.8 and the gradients of 16 workers
// of 500 181.5; now 28.9, 123.3 and 178.4.
template <bool kTwo>
__global__ void __launch_bounds__(128) logits_loss_kernel(int C, int K, int B, int rows_cta,
                                                          const float* __restrict__ A, const float* __restrict__ pool,
                                                          const int32_t* __restrict__ idx, int64_t S,
                                                          const int32_t* __restrict__ labels,
                                                          const float* __restrict__ W, const float* __restrict__ bias,
                                                          float* __restrict__ sample_loss, float* __restrict__ dZ,
                                                          float* __restrict__ loss, int* __restrict__ cnt) {
    grid_begin();
    const int i = blockIdx.y, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t row0 = (int64_t)i * B;
    const int rbeg = blockIdx.x * rows_cta, rend = rbeg + rows_cta < B ? rbeg + rows_cta : B;
    const float invB = 1.0f / static_cast<float>(B);
    for (int r = rbeg + warp; r < rend; r += 4) {
        const int64_t m = row0 + r, sidx = idx[m];
        const bool in = sidx >= 0 && sidx < S;
        const int y = in ? labels[sidx] : -1;
        const bool bad = y < 0 || y >= C;
        const float* a = pool ? pool + (in ? sidx : 0) * K : A + m * K;
        const float dot = skinny_row<kTwo>(a, W, K, C, K, lane);
        const float z = lane < C ? dot + bias[lane] : -INFINITY;
        float mx = z;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
        const float ez = lane < C ? expf(z - mx) : 0.f;
        float se = ez;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) se += __shfl_xor_sync(0xffffffffu, se, o);
        const float inv_se = 1.0f / se, zy = __shfl_sync(0xffffffffu, z, y & 31);
        float g = ez * inv_se;
        if (lane == y) g -= 1.0f;
        if (lane < C) dZ[m * C + lane] = bad ? NAN : g * invB;
        if (lane == 0) sample_loss[m] = bad ? NAN : (mx + logf(se)) - zy;
    }
    finish_worker_loss<128>(sample_loss + row0, B, gridDim.x, cnt + i, invB, loss + i);
}

// Input-gradient GEMM with a short inner dimension (K = out <= kSkinnyK):
// dZ_{l-1}[m, c] = (sum_{o < K} dZ_l[m, o] W[o, c]) * 1[act[m, c] > 0], the products
// added in increasing o (EpiDx's arithmetic, with the 16 masks loaded before any
// store).  W and the CTA's 16 rows of dZ_l sit in shared memory; a thread per column
// computes the 16 rows' outputs.  With ``hiT`` it also writes their tf32 parts transposed, as
// split_t_kernel would from dZ_{l-1} (hiT / loT [N, ldt], workers of B samples in blocks of
// B + pad columns): with that pass apart, and the gather's rows loaded one after another,
// 784-256-10 took 122.6 us an iteration at 64 workers of 64 samples and 179.4 for the gradients of
// 16 of 500; now 118.4 and 173.7 (with 16-byte stores of the parts 120.1 and 176.4).
template <typename T>
__global__ void __launch_bounds__(256) skinny_k_dx_kernel(int M, int N, int K, const T* __restrict__ dZ, int64_t ldz,
                                                          const T* __restrict__ W, int64_t ldw, EpiDx<T> epi,
                                                          float* __restrict__ hiT, float* __restrict__ loT, int64_t ldt,
                                                          int B, int pad) {
    grid_begin();
    constexpr int R = 16;                               // rows per CTA
    extern __shared__ float wsh[];                      // W as [K, N] fp32, then the CTA's dZ rows [R, K]
    float* zsh = wsh + N * K;
    fill_shared(wsh, N * K, [&](int e) { return to_f(W[(int64_t)(e / N) * ldw + e % N]); });
    for (int m0 = blockIdx.y * R; m0 < M; m0 += gridDim.y * R) {
        __syncthreads();   // the previous rows' reads of zsh are done
        fill_shared(zsh, R * K, [&](int e) {
            const int m = m0 + e / K;
            return m < M ? to_f(dZ[(int64_t)m * ldz + e % K]) : 0.f;
        });
        __syncthreads();
        for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < N; c += gridDim.x * blockDim.x) {
            float v[R];
#pragma unroll
            for (int j = 0; j < R; ++j) v[j] = 0.f;
            for (int o = 0; o < K; ++o) {
                const float wv = wsh[o * N + c];
#pragma unroll
                for (int j = 0; j < R; ++j) v[j] = fmaf(zsh[j * K + o], wv, v[j]);
            }
            // the ReLU masks of the R rows, all loaded before the first store
            float a[R];
#pragma unroll
            for (int j = 0; j < R; ++j) a[j] = m0 + j < M ? to_f(epi.act[(int64_t)(m0 + j) * epi.ldo + c]) : 0.f;
#pragma unroll
            for (int j = 0; j < R; ++j) {
                v[j] = v[j] * (a[j] > 0.f ? 1.f : 0.f);
                if (m0 + j < M) epi.out[(int64_t)(m0 + j) * epi.ldo + c] = from_f<T>(v[j]);
            }
            if (hiT) {
                float* hp = hiT + (int64_t)c * ldt;
                float* lp = loT + (int64_t)c * ldt;
                if (pad == 0 && ldt % 8 == 0 && m0 + R <= M) {   // whole 32-byte sectors
#pragma unroll
                    for (int j = 0; j < R; j += 8) {
                        uint32_t h[8], l[8];
#pragma unroll
                        for (int q = 0; q < 8; ++q) {
                            float x, y;
                            tf32::split_value(v[j + q], x, y);
                            h[q] = __float_as_uint(x);
                            l[q] = __float_as_uint(y);
                        }
                        tcx::store_256(hp + m0 + j, h);
                        tcx::store_256(lp + m0 + j, l);
                    }
                } else {
                    for (int j = 0; j < R && m0 + j < M; ++j) {
                        const int t = m0 + j + (m0 + j) / B * pad;
                        float h, l;
                        tf32::split_value(v[j], h, l);
                        hp[t] = h;
                        lp[t] = l;
                    }
                }
            }
        }
    }
}

// Weight gradient of a layer with few outputs (out <= kSkinnyN, the logits layer):
// G[i, offW + o in + c] = sum_{r < B} dZ[i B + r, o] A[i B + r, c], and the bias part, its sum
// over the rows of dZ alone.  CTA = 32 columns of one worker: the dZ rows sit in shared
// memory kDwRows at a time (padded to 4 NO4 outputs), A's row numbers beside them (the stacked
// rows, or with ``idx`` the samples' rows of the pool; outside [0, S): row 0), warp w of nw takes rows w, w + nw, .. with its
// 8 next activations loaded at a time (nw = 8, fewer below 32 rows: at least four rows a warp, whose
// products are not rounded apart), and the warps' sums are added in warp order; the first
// column block also adds the bias part.  (On 128 x 128 FFMA tiles 118 of 128 rows were padding
// and a CTA ran all B rows alone: 9.8 us for 64 workers of 64 samples, 256 x 10, and 5.4 for 16
// of 32, 784 x 10, beside bias launches of 3.6 and 1.8; here 4.9 and under 3 with the bias.)
constexpr int kDwRows = 128;
template <typename T, int NO4>
__global__ void __launch_bounds__(256) skinny_dw_kernel(const T* __restrict__ dZ, const T* __restrict__ A,
                                                        const int32_t* __restrict__ idx, int64_t S, int out, int in,
                                                        int B, float* __restrict__ G, int64_t ldG, int64_t offW,
                                                        int64_t offb) {
    grid_begin();
    constexpr int NO = 4 * NO4;
    __shared__ __align__(16) float zs[kDwRows][NO];
    __shared__ float red[8][NO][33];
    const int i = blockIdx.y, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int c = blockIdx.x * 32 + lane;
    const T* z = dZ + (int64_t)i * B * out;
    __shared__ int src[kDwRows];   // row of A of each of the rows
    const T* a = A + c;
    float acc[NO];
#pragma unroll
    for (int o = 0; o < NO; ++o) acc[o] = 0.f;
    float bsum = 0.f;   // bias: output threadIdx.x % NO, rows threadIdx.x / NO, + 256 / NO, ..
    for (int r0 = 0; r0 < B; r0 += kDwRows) {
        const int rows = B - r0 < kDwRows ? B - r0 : kDwRows;
        __syncthreads();   // the previous rows' reads of zs are done
        for (int e = threadIdx.x; e < rows * NO; e += 256) {
            const int r = e / NO, o = e % NO;
            zs[r][o] = o < out ? to_f(z[(int64_t)(r0 + r) * out + o]) : 0.f;
        }
        for (int r = threadIdx.x; r < rows; r += 256) {
            const int m = i * B + r0 + r;   // M = n B < 2^31
            src[r] = m;
            if (idx) {
                const int64_t q = idx[m];
                src[r] = q >= 0 && q < S ? static_cast<int>(q) : 0;
            }
        }
        __syncthreads();
        const int nw = rows >= 32 ? 8 : rows >= 8 ? rows / 4 : 1;
        for (int q0 = warp < nw ? warp : rows; q0 < rows; q0 += 8 * nw) {
            float av[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const int r = q0 + nw * u;
                av[u] = r < rows && c < in ? to_f(a[(int64_t)src[r] * in]) : 0.f;
            }
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const int r = q0 + nw * u;
                if (r >= rows) break;
#pragma unroll
                for (int g = 0; g < NO4; ++g) {
                    const float4 zv = *reinterpret_cast<const float4*>(&zs[r][4 * g]);
                    acc[4 * g] = fmaf(zv.x, av[u], acc[4 * g]);
                    acc[4 * g + 1] = fmaf(zv.y, av[u], acc[4 * g + 1]);
                    acc[4 * g + 2] = fmaf(zv.z, av[u], acc[4 * g + 2]);
                    acc[4 * g + 3] = fmaf(zv.w, av[u], acc[4 * g + 3]);
                }
            }
        }
        if (blockIdx.x == 0)
            for (int r = threadIdx.x / NO; r < rows; r += 256 / NO) bsum += zs[r][threadIdx.x % NO];
    }
#pragma unroll
    for (int o = 0; o < NO; ++o) red[warp][o][lane] = acc[o];
    __syncthreads();
    float* g = G + (int64_t)i * ldG;
    for (int e = threadIdx.x; e < out * 32; e += 256) {
        const int o = e >> 5;
        float t = 0.f;
#pragma unroll
        for (int w = 0; w < 8; ++w) t += red[w][o][lane];
        if (c < in) g[offW + (int64_t)o * in + c] = t;
    }
    if (blockIdx.x == 0) {
        float* bs = &zs[0][0];   // 256 partial sums (zs holds at least 512 floats)
        __syncthreads();
        bs[threadIdx.x] = bsum;
        __syncthreads();
        if (threadIdx.x < out) {
            float t = 0.f;
            for (int q = 0; q < 256 / NO; ++q) t += bs[q * NO + threadIdx.x];
            g[offb + threadIdx.x] = t;
        }
    }
}

template <typename T>
cudaError_t launch_skinny_dw(const T* dZ, const T* A, const int32_t* idx, int64_t S, int out, int in, int n,
                             int B, float* G, int64_t ldG, int64_t offW, int64_t offb, cudaStream_t st) {
    const dim3 grid((in + 31) / 32, n);
    auto kern = out <= 4 ? skinny_dw_kernel<T, 1> : out <= 8 ? skinny_dw_kernel<T, 2> : skinny_dw_kernel<T, 4>;
    launch(kern, grid, 256, 0, st, dZ, A, idx, S, out, in, B, G, ldG, offW, offb);
    return cudaGetLastError();
}

inline bool skinny_n_ok(int N, int K) { return N <= kSkinnyN && (size_t)N * K * 4 <= kSkinnySmem; }
inline bool skinny_k_ok(int N, int K) { return K <= kSkinnyK && ((size_t)N + 16) * K * 4 <= kSkinnySmem; }

template <typename T, bool A_K, bool B_K, class Epi>
cudaError_t run_gemm(int M, int N, int K, const T* A, int64_t lda, int64_t batchA, const T* B, int64_t ldb,
                     int64_t batchB, int batch, Epi epi, cudaStream_t st, float* split_ws = nullptr,
                     size_t split_floats = 0) {
    int splits = split_ws ? splitk_count(M, N, K, batch) : 1;
    while (splits > 1 && (size_t)splits * M * N > split_floats) --splits;
    if (splits > 1) {
        const int kps = ((K + splits - 1) / splits + BK - 1) / BK * BK;
        splits = (K + kps - 1) / kps;
        dim3 grid((N + BN - 1) / BN, (M + BM - 1) / BM, splits);
        launch(gemm_simt_kernel<T, A_K, B_K, Epi, true>, grid, 256, 0, st, M, N, K, A, lda, 0, B, ldb, 0, epi, kps,
                                                                       split_ws);
        const int64_t total = (int64_t)M * N;
        const int blocks = static_cast<int>((total + 255) / 256 < 4 * sm_count() ? (total + 255) / 256 : 4 * sm_count());
        launch(splitk_reduce_kernel<Epi>, blocks, 256, 0, st, M, N, splits, split_ws, epi);
        return cudaGetLastError();
    }
    dim3 grid((N + BN - 1) / BN, (M + BM - 1) / BM, batch);
    launch(gemm_simt_kernel<T, A_K, B_K, Epi, false>, grid, 256, 0, st, M, N, K, A, lda, batchA, B, ldb, batchB, epi, K,
                                                                    nullptr);
    return cudaGetLastError();
}

// T: the operand type.  The tf32 and 16-byte kernels serve fp32 alone.
template <typename T>
int worker_grads_simt(const GradsPlan& P, const float* w, const float* pool, int64_t S, const int32_t* labels,
                      const int32_t* idx, float* G, int64_t ld, float* loss, char* ws, cudaStream_t st) {
    const int L = P.L;
    const int M = P.M;
    const int B = P.B;
    constexpr bool kF32 = sizeof(T) == 4;
    T* X = reinterpret_cast<T*>(ws + P.off_x);
    float* logits = reinterpret_cast<float*>(ws + P.off_logits);
    float* sloss = reinterpret_cast<float*>(ws + P.off_sloss);
    T* dz[2] = {reinterpret_cast<T*>(ws + P.off_dz[0]), reinterpret_cast<T*>(ws + P.off_dz[1])};
    float* split_ws = P.split_floats ? reinterpret_cast<float*>(ws + P.off_split) : nullptr;
    // the status word and the workers' loss counters
    const bool parts = P.tf32[0] || P.tf32_dw[0];   // the gather writes the first layer's tf32 parts
    if (!parts) {
        const cudaError_t e0 = cudaMemsetAsync(ws, 0, P.off_cnt + P.n * sizeof(int), st);
        if (e0 != cudaSuccess) return fail(DBW_ECUDA, "dbw_worker_grads: %s", cudaGetErrorString(e0));
    }
    const T* wop;   // the weights as operands
    if constexpr (kF32) {
        wop = w;
    } else {
        launch(cast_bf16_kernel, 4 * sm_count(), 256, 0, st, w, P.d, reinterpret_cast<T*>(ws + P.off_wb));
        wop = reinterpret_cast<const T*>(ws + P.off_wb);
    }
    // the last layer's logits, loss and dZ_L in one launch; a single layer then needs no gather
    const bool few = kF32 && P.widths[L] <= kSkinnyN && P.widths[L - 1] % 4 == 0 && aligned16(w + P.offW[L - 1]);
    const bool from_pool = few && L == 1;
    if (!from_pool) {
        const int in = P.widths[0];
        if (parts) {
            // the first layer's GEMMs in three tf32 passes take their X parts from the gather;
            // X itself only when one of them stays on SIMT
            const int gx = (in + 127) / 128, ty = (M + 31) / 32 < 60000 ? (M + 31) / 32 : 60000;
            // the weights: up to 4 CTAs per SM (in % 4 == 0 and w is 16-byte aligned: a flat pass)
            const int64_t nw4 = P.tf32[0] ? (int64_t)P.widths[1] * in / 4 : 0;
            const int64_t wc = (nw4 + 255) / 256 < 4 * sm_count() ? (nw4 + 255) / 256 : 4 * sm_count();
            const int wy = static_cast<int>((wc + gx - 1) / gx);
            const bool need_x = !(P.tf32[0] && P.tf32_dw[0]);
            launch(gather_parts_kernel, dim3(gx, ty + wy), dim3(32, 8), 0, st, ty, w + P.offW[0], nw4,
                reinterpret_cast<float*>(ws + P.off_whi), reinterpret_cast<float*>(ws + P.off_wlo),
                reinterpret_cast<int*>(ws), static_cast<int>(P.off_cnt / 4) + P.n, pool, S, in, idx, M, need_x ? reinterpret_cast<float*>(X) : nullptr,
                P.tf32[0] ? reinterpret_cast<float*>(ws + P.off_ahi) : nullptr,
                P.tf32[0] ? reinterpret_cast<float*>(ws + P.off_alo) : nullptr, (in + 3) / 4 * 4,
                P.tf32_dw[0] ? reinterpret_cast<float*>(ws + P.off_xthi) : nullptr,
                P.tf32_dw[0] ? reinterpret_cast<float*>(ws + P.off_xtlo) : nullptr, P.n * tf32::padded_samples(B), B,
                static_cast<int>(tf32::padded_samples(B) - B));
        } else {
            launch(gather_kernel<T>, dim3((in + 1023) / 1024, M < 65535 ? M : 65535), 256, 0, st, pool, S, in, idx, M, X);
        }
    }
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return fail(DBW_ECUDA, "gather launch: %s", cudaGetErrorString(e));

    // forward
    const T* Ain = X;
    for (int l = 0; l < L; ++l) {
        const int fin = P.widths[l], fout = P.widths[l + 1];
        const T* W = wop + P.offW[l];
        const float* bias = w + P.offb[l];
        const bool tc = P.tf32[l];
        float* part[4] = {nullptr, nullptr, nullptr, nullptr};
        if (tc) {
            part[0] = reinterpret_cast<float*>(ws + P.off_ahi);
            part[1] = reinterpret_cast<float*>(ws + P.off_alo);
            part[2] = reinterpret_cast<float*>(ws + P.off_whi);
            part[3] = reinterpret_cast<float*>(ws + P.off_wlo);
        }
        int* status = reinterpret_cast<int*>(ws);
        auto fwd = [&](auto epi) {
            if constexpr (kF32) {
                if (tc)
                    return tf32::run(M, fout, fin, Ain, fin, W, fin, part[0], part[1], part[2], part[3], epi, status, st,
                                     /*parts_ready=*/l == 0);
                // (the last layer's go to logits_loss_kernel)
                if constexpr (!std::is_same<decltype(epi), EpiLogits>::value) {
                    if (fout <= kSkinnyN && fin % 4 == 0 && aligned16(Ain) && aligned16(W)) {
                        const int want = (M + 3) / 4;   // 4 rows (warps) per CTA
                        const int grid = want < 8 * sm_count() ? want : 8 * sm_count();
                        auto kern = fin > 256 ? skinny_n4_kernel<true, decltype(epi)> : skinny_n4_kernel<false, decltype(epi)>;
                        launch(kern, grid, 128, 0, st, M, fout, fin, Ain, fin, W, fin, epi);
                        return cudaGetLastError();
                    }
                }
            }
            if (skinny_n_ok(fout, fin)) {
                const int rows_per_cta = 8;
                const int want = (M + rows_per_cta - 1) / rows_per_cta;
                const int grid = want < 2 * sm_count() ? want : 2 * sm_count();
                launch(skinny_n_kernel<T, decltype(epi)>, grid, 256, (size_t)fout * fin * 4, st, M, fout, fin, Ain, fin, W, fin, epi);
                return cudaGetLastError();
            }
            return run_gemm<T, true, true>(M, fout, fin, Ain, fin, 0, W, fin, 0, 1, epi, st, split_ws, P.split_floats);
        };
        if (l < L - 1) {
            T* Aout = reinterpret_cast<T*>(ws + P.off_act[l + 1]);
            e = fwd(EpiHidden<T>{bias, Aout, fout});
            Ain = Aout;
        } else {
            if (few) break;
            e = fwd(EpiLogits{bias, logits, fout});
        }
        if (e != cudaSuccess) return fail(DBW_ECUDA, "forward GEMM %d: %s", l, cudaGetErrorString(e));
    }
    const int C = P.widths[L];
    if (few) {
        if constexpr (kF32) {
            const int fin = P.widths[L - 1];
            // 4 rows (a warp each) per CTA, or as many fours as bring the grid to 8 CTAs per SM
            const int64_t most = 8 * sm_count();
            const int rows_cta = static_cast<int>(4 * (((M + 3) / 4 + most - 1) / most));
            const dim3 grid((B + rows_cta - 1) / rows_cta, P.n);
            launch(fin > 256 ? logits_loss_kernel<true> : logits_loss_kernel<false>, grid, 128, 0, st, C, fin, B, rows_cta,
                   Ain, from_pool ? pool : nullptr, idx, S, labels, w + P.offW[L - 1], w + P.offb[L - 1], sloss, dz[0], loss,
                   reinterpret_cast<int*>(ws + P.off_cnt));
            e = cudaGetLastError();
        }
    } else
        e = launch_softmax(logits, C, C, P.n, B, idx, S, labels, sloss, dz[0], C, loss,
                           reinterpret_cast<int*>(ws + P.off_cnt), st);
    if (e != cudaSuccess) return fail(DBW_ECUDA, "loss launch: %s", cudaGetErrorString(e));

    // backward
    int cur = 0;
    bool dz_parts_ready = false;   // dZ_l's transposed parts are in the workspace
    for (int l = L - 1; l >= 0; --l) {
        const int fin = P.widths[l], fout = P.widths[l + 1];
        const T* Aprev = (l == 0) ? X : reinterpret_cast<const T*>(ws + P.off_act[l]);
        const T* dZl = dz[cur];
        // per-worker weight gradient: M' = fout, N' = fin, K = B; A(o, r) = dZ[r*fout + o], B(r, c) = A[r*fin + c]
        if (fout <= kSkinnyN) {
            const T* rows = Aprev;
            if constexpr (kF32) rows = from_pool ? pool : Aprev;
            e = launch_skinny_dw(dZl, rows, from_pool ? idx : nullptr, S, fout, fin, P.n, B, G, ld, P.offW[l], P.offb[l], st);
        } else if (P.tf32_dw[l]) {
            const size_t ath = l == 0 ? P.off_xthi : P.off_athi, atl = l == 0 ? P.off_xtlo : P.off_atlo;
            if constexpr (kF32)
                e = tf32::run_dw(fout, fin, B, P.n, dZl, fout, Aprev, fin, reinterpret_cast<float*>(ws + P.off_zthi),
                                 reinterpret_cast<float*>(ws + P.off_ztlo), reinterpret_cast<float*>(ws + ath),
                                 reinterpret_cast<float*>(ws + atl), G + P.offW[l], fin, ld, reinterpret_cast<int*>(ws),
                                 st, /*act_parts_ready=*/l == 0, dz_parts_ready);
        } else {
            e = run_gemm<T, false, false>(fout, fin, B, dZl, fout, (int64_t)B * fout, Aprev, fin, (int64_t)B * fin, P.n,
                                       EpiDW{G, ld, P.offW[l], fin}, st);
        }
        if (e != cudaSuccess) return fail(DBW_ECUDA, "dW GEMM %d: %s", l, cudaGetErrorString(e));
        dz_parts_ready = false;
        if (fout > kSkinnyN) e = launch_bias_grad(dZl, fout, fout, P.n, B, G, ld, P.offb[l], st);
        if (e != cudaSuccess) return fail(DBW_ECUDA, "bias grad %d: %s", l, cudaGetErrorString(e));
        if (l > 0) {
            // dZ_{l-1}[m, c] = sum_o dZ_l[m, o] W_l[o, c]: A(m, o) = dZ[m*fout + o], B(o, c) = W[o*fin + c]
            T* dnext = dz[cur ^ 1];
            if (skinny_k_ok(fin, fout)) {
                const int ry = (M + 15) / 16;
                dim3 grid((fin + 255) / 256, ry < 65535 ? ry : 65535);
                const bool parts = P.tf32_dw[l - 1];   // the next weight gradient reads the transposed parts
                const int Kp = static_cast<int>(tf32::padded_samples(B));
                launch(skinny_k_dx_kernel<T>, grid, 256, ((size_t)fin + 16) * fout * 4, st, M, fin, fout, dZl, fout,
                       wop + P.offW[l], fin, EpiDx<T>{Aprev, dnext, fin},
                       parts ? reinterpret_cast<float*>(ws + P.off_zthi) : nullptr,
                       parts ? reinterpret_cast<float*>(ws + P.off_ztlo) : nullptr, (int64_t)P.n * Kp, B, Kp - B);
                dz_parts_ready = parts;
                e = cudaGetLastError();
            } else {
                e = run_gemm<T, true, false>(M, fin, fout, dZl, fout, 0, wop + P.offW[l], fin, 0, 1,
                                             EpiDx<T>{Aprev, dnext, fin}, st, split_ws, P.split_floats);
            }
            if (e != cudaSuccess) return fail(DBW_ECUDA, "dX GEMM %d: %s", l, cudaGetErrorString(e));
            cur ^= 1;
        }
    }
    return DBW_OK;
}

}  // namespace

bool make_grads_plan(int L, const int32_t* widths, int n, int B, int prec, GradsPlan* P) {
    if (L < 1 || L > DBW_LMAX || n < 1 || n > DBW_NMAX || B < 1) return false;
    if (prec != DBW_PREC_FP32 && prec != DBW_PREC_BF16) return false;
    P->L = L;
    P->n = n;
    P->B = B;
    P->prec = prec;
    const int64_t M = (int64_t)n * B;
    if (M > (1LL << 30)) return false;
    P->M = (int)M;
    int maxw = 0;
    int64_t off = 0;
    for (int l = 0; l <= L; ++l) {
        if (widths[l] < 1 || widths[l] > (1 << 20)) return false;
        P->widths[l] = widths[l];
        if (l > 0 && widths[l] > maxw) maxw = widths[l];   // of the layers dZ is formed for
    }
    if (widths[L] < 2) return false;
    for (int l = 0; l < L; ++l) {
        P->offW[l] = off;
        off += (int64_t)widths[l + 1] * widths[l];
        P->offb[l] = off;
        off += widths[l + 1];
    }
    P->d = off;
    size_t cur = 0;
    auto take = [&](size_t bytes) {
        const size_t at = cur;
        cur += (bytes + 255) / 256 * 256;
        return at;
    };
    take(256);   // status word (int32 at offset 0), as in the tcgen05 plan
    P->off_cnt = take((size_t)n * 4);
    const size_t es = prec == DBW_PREC_BF16 ? 2 : 4;
    P->off_x = take((size_t)M * widths[0] * es);
    P->off_act[0] = P->off_x;
    for (int l = 1; l < L; ++l) P->off_act[l] = take((size_t)M * widths[l] * es);
    P->off_logits = take((size_t)M * widths[L] * 4);
    P->off_sloss = take((size_t)M * 4);
    P->off_dz[0] = take((size_t)M * maxw * es);
    P->off_dz[1] = take((size_t)M * maxw * es);
    P->off_wb = prec == DBW_PREC_BF16 ? take((size_t)P->d * 2) : 0;
    // split-K scratch of the forward and input-gradient GEMMs (the largest splits x M x N)
    size_t split = 0;
    for (int l = 0; l < L; ++l) {
        const int fin = widths[l], fout = widths[l + 1];
        const size_t f = (size_t)splitk_count(P->M, fout, fin, 1) * P->M * fout;
        const size_t x = l > 0 ? (size_t)splitk_count(P->M, fin, fout, 1) * P->M * fin : 0;
        split = f > split ? f : split;
        split = x > split ? x : split;
    }
    P->split_floats = split;
    P->off_split = split ? take(split * 4) : 0;
    // forward GEMMs with at least 2^27 multiply-adds and 32 outputs run in three tf32 passes
    size_t a_parts = 0, w_parts = 0;
    for (int l = 0; l < L; ++l) {
        const int fin = widths[l], fout = widths[l + 1];
        P->tf32[l] = prec == DBW_PREC_FP32 && fout >= 32 && (int64_t)P->M * fout * fin >= (int64_t(1) << 27);
        if (!P->tf32[l]) continue;
        const size_t ld4 = (size_t)(fin + 3) / 4 * 4;
        a_parts = (size_t)P->M * ld4 > a_parts ? (size_t)P->M * ld4 : a_parts;
        w_parts = (size_t)fout * ld4 > w_parts ? (size_t)fout * ld4 : w_parts;
    }
    P->off_ahi = a_parts ? take(a_parts * 4) : 0;
    P->off_alo = a_parts ? take(a_parts * 4) : 0;
    P->off_whi = w_parts ? take(w_parts * 4) : 0;
    P->off_wlo = w_parts ? take(w_parts * 4) : 0;
    // weight gradients with at least 2^25 multiply-adds run in three tf32 passes when the G
    // rows of the layer take 16-byte stores (a ragged B up to 128: less exact than FFMA, see dw_kernel)
    const size_t Mt = (size_t)n * tf32::padded_samples(B);   // columns of the transposed parts
    size_t zt = 0, at = 0;
    for (int l = 0; l < L; ++l) {
        const int fin = widths[l], fout = widths[l + 1];
        P->tf32_dw[l] = prec == DBW_PREC_FP32 && (B % 32 == 0 || B > 128) && fin % 4 == 0 &&
                        P->offW[l] % 4 == 0 && fout >= 32 && (int64_t)n * fout * fin * B >= (int64_t(1) << 25);
        if (!P->tf32_dw[l]) continue;
        zt = (size_t)fout * Mt > zt ? (size_t)fout * Mt : zt;
        if (l > 0) at = (size_t)fin * Mt > at ? (size_t)fin * Mt : at;
    }
    P->off_zthi = zt ? take(zt * 4) : 0;
    P->off_ztlo = zt ? take(zt * 4) : 0;
    P->off_athi = at ? take(at * 4) : 0;
    P->off_atlo = at ? take(at * 4) : 0;
    const size_t xt = P->tf32_dw[0] ? (size_t)widths[0] * Mt : 0;
    P->off_xthi = xt ? take(xt * 4) : 0;
    P->off_xtlo = xt ? take(xt * 4) : 0;
    P->ws_bytes = cur;
    return true;
}

int grads_activations(int L, const int32_t* widths, int n, int B, int prec, int layer, size_t* offset, int64_t* ld,
                      int* elem_bytes) {
    if (layer < 1 || layer >= L) return fail(DBW_EINVAL, "dbw_worker_grads_activations: layer must be in [1, L-1]");
    if (tc_eligible(prec, L, B)) {
        TcPlan T;
        if (!make_tc_plan(L, widths, n, B, &T)) return fail(DBW_EINVAL, "dbw_worker_grads_activations: invalid shape");
        *offset = T.off_act[layer];
        *ld = T.ldact[layer];
        *elem_bytes = 2;
        return DBW_OK;
    }
    GradsPlan P;
    if (!make_grads_plan(L, widths, n, B, prec, &P)) return fail(DBW_EINVAL, "dbw_worker_grads_activations: invalid shape");
    *offset = P.off_act[layer];
    *ld = widths[layer];
    *elem_bytes = prec == DBW_PREC_BF16 ? 2 : 4;
    return DBW_OK;
}

size_t grads_workspace_bytes(int L, const int32_t* widths, int n, int B, int prec) {
    if (tc_eligible(prec, L, B)) {
        TcPlan T;
        if (!make_tc_plan(L, widths, n, B, &T)) return 0;
        return T.ws_bytes;
    }
    GradsPlan P;
    if (!make_grads_plan(L, widths, n, B, prec, &P)) return 0;
    return P.ws_bytes;
}

int launch_worker_grads(int L, const int32_t* widths, int prec, const float* w, int64_t d, const float* pool,
                        int64_t S, const int32_t* labels, const int32_t* idx, int n, int B, float* G, int64_t ld,
                        float* loss, void* ws, size_t ws_bytes, cudaStream_t st) {
    GradsPlan P;
    if (!make_grads_plan(L, widths, n, B, prec, &P)) return fail(DBW_EINVAL, "dbw_worker_grads: invalid model shape");
    if (P.d != d) return fail(DBW_EINVAL, "dbw_worker_grads: d = %lld but the widths give %lld", (long long)d,
                              (long long)P.d);
    if (tc_eligible(prec, L, B)) {
        TcPlan T;
        if (!make_tc_plan(L, widths, n, B, &T)) return fail(DBW_EINVAL, "dbw_worker_grads: invalid model shape");
        if (ws_bytes < T.ws_bytes)
            return fail(DBW_EINVAL, "dbw_worker_grads: workspace %zu bytes < %zu needed", ws_bytes, T.ws_bytes);
        return worker_grads_tc(T, w, pool, S, labels, idx, G, ld, loss, static_cast<char*>(ws), st);
    }
    if (ws_bytes < P.ws_bytes)
        return fail(DBW_EINVAL, "dbw_worker_grads: workspace %zu bytes < %zu needed", ws_bytes, P.ws_bytes);
    if (prec == DBW_PREC_BF16)
        return worker_grads_simt<__nv_bfloat16>(P, w, pool, S, labels, idx, G, ld, loss, static_cast<char*>(ws), st);
    return worker_grads_simt<float>(P, w, pool, S, labels, idx, G, ld, loss, static_cast<char*>(ws), st);
}

}  // namespace dbw
