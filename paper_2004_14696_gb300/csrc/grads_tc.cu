// Eq. (2) for all n workers with bf16 GEMM operands on the tcgen05 tensor cores.
//
// Same computation as the fp32 pass in grads.cu (forward over the stacked
// M = n B rows, softmax cross entropy, backward with a per-worker weight
// gradient of depth K = B) on the GEMMs of gemm_tc.cu:
//
//   forward   Z_l = A_{l-1} . W_l^T          A = act[l-1] [M, in],   B = W_l [out, in]
//   dX        dZ_{l-1} = dZ_l . W_l          A = dZ_l [M, out],      B = W_l [out, in]
//   dW        G_i = dZ_l[i]^T . A_{l-1}[i]   A = dZ_l [M, out],      B = act[l-1] [M, in]
//                                            (worker i: rows i*B .. i*B+B-1, K = B)
//
// A worker's rows are read through a 3-D tensor map (column, sample, worker), so the last K
// block of a B that is not whole K blocks reads zeros past the worker's samples (tc_eligible says
// which such B run here).
//
// Every operand is the row-major bf16 buffer its producer wrote: the tensor cores read
// dZ, the activations and (in dX) W as MN-major tiles, so no transposed copy is formed.
// With transposed copies (written by the GEMM epilogues, the X and W casts and the
// softmax; a third of the casts' bytes and half of the epilogues' stores) the
// 3072-1024-1024-10 pass of 128 x 128 samples took 822 us, without them 734.
// Leading dimensions are padded to multiples of 8 elements (16 bytes, the TMA
// stride rule); tensor maps carry the logical extents, and the bias sums, whose 16-byte
// loads reach into the padding, drop its columns.
#include <math.h>

#include "gemm_tc.cuh"
#include "grads.cuh"
#include "loss_bias.cuh"
#include "tc_ptx.cuh"

namespace dbw {

namespace {

inline int64_t rup(int64_t x, int64_t m) { return (x + m - 1) / m * m; }

// out[m, :] = bf16(src[row(m), :]) for one row of ``cols`` values, by one warp: a lane
// takes groups of 8 columns (two 16-byte loads, one 16-byte store), four groups' loads in
// flight.  src rows are 16-byte aligned when ``vec``; ldo is a multiple of 8.
__device__ __forceinline__ void cast_row(const float* __restrict__ s, int cols, __nv_bfloat16* __restrict__ o,
                                         bool vec) {
    const int lane = threadIdx.x & 31;
    const int groups = vec ? cols / 8 : 0;
    for (int g0 = lane; g0 < groups; g0 += 128) {
        float4 v[4][2];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int g = g0 + 32 * u;
            if (g < groups) {
                v[u][0] = __ldcs(reinterpret_cast<const float4*>(s) + 2 * g);
                v[u][1] = __ldcs(reinterpret_cast<const float4*>(s) + 2 * g + 1);
            }
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int g = g0 + 32 * u;
            if (g < groups) {
                uint4 h;
                h.x = tcx::pack_bf16(v[u][0].x, v[u][0].y);
                h.y = tcx::pack_bf16(v[u][0].z, v[u][0].w);
                h.z = tcx::pack_bf16(v[u][1].x, v[u][1].y);
                h.w = tcx::pack_bf16(v[u][1].z, v[u][1].w);
                reinterpret_cast<uint4*>(o)[g] = h;
            }
        }
    }
    for (int c = 8 * groups + lane; c < cols; c += 32) o[c] = __float2bfloat16_rn(s[c]);
}

// X: out[m, :] = bf16(src[rowmap(m), :]) for the live rows; rowmap(m) < 0 makes row m
// zero.  A warp per row, grid-stride.  The pool's rows are 16-byte aligned (the width is
// a multiple of 4 and the base aligned: checked by the caller).
template <class RowMap>
__global__ void __launch_bounds__(256) cast_rows_kernel(const float* __restrict__ src, int64_t lds, int rows, int cols,
                                                        RowMap rowmap, __nv_bfloat16* __restrict__ out, int64_t ldo) {
    grid_begin();
    const int live = rowmap.live(rows);
    const int warps = gridDim.x * (blockDim.x >> 5);
    for (int m = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; m < live; m += warps) {
        const int64_t sr = rowmap(m);
        __nv_bfloat16* o = out + static_cast<int64_t>(m) * ldo;
        if (sr >= 0) {
            cast_row(src + sr * lds, cols, o, true);
        } else {
            for (int c = threadIdx.x & 31; c < cols; c += 32) o[c] = __float2bfloat16_rn(0.f);
        }
    }
}

// Every layer's W_l -> bf16 in one launch: a warp per row, the layers' rows one after the
// other (r0: first row of layer l).
struct WeightCasts {
    int L;
    const float* w[DBW_LMAX];
    int fin[DBW_LMAX];
    int r0[DBW_LMAX + 1];
    bool vec[DBW_LMAX];       // rows of W_l 16-byte aligned
    __nv_bfloat16* wb[DBW_LMAX];
    int64_t ldw[DBW_LMAX];
};

__global__ void __launch_bounds__(256) cast_weights_kernel(WeightCasts a) {
    grid_begin();
    const int warps = gridDim.x * (blockDim.x >> 5);
    for (int r = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; r < a.r0[a.L]; r += warps) {
        int l = 0;
        while (l + 1 < a.L && r >= a.r0[l + 1]) ++l;
        const int64_t o = r - a.r0[l];
        cast_row(a.w[l] + o * a.fin[l], a.fin[l], a.wb[l] + o * a.ldw[l], a.vec[l]);
    }
}

struct GatherRows {     // X of the per-worker pass: pool row idx[m]; an index outside [0, S) reads row 0
    const int32_t* idx;
    int64_t S;
    __device__ int live(int rows) const { return rows; }
    __device__ int64_t operator()(int m) const {
        const int64_t r = idx[m];
        return (r < 0 || r >= S) ? 0 : r;
    }
};

// X of the received-workers pass: row m of slot s = m / B < k is pool row
// idx[sel[s] B + m % B] (an index outside [0, S) reads row 0); rows from k B up to
// the live row count are zero; later rows are not written.
struct ReceivedRows {
    const int32_t* idx;
    const int32_t* sel;
    const int* kdev;
    int B;
    int64_t S;
    __device__ int live(int rows) const { return live_rows(kdev, B, rows); }
    __device__ int64_t operator()(int m) const {
        const int s = m / B;
        if (s >= *kdev) return -1;
        const int64_t r = idx[static_cast<int64_t>(sel[s]) * B + (m - s * B)];
        return (r < 0 || r >= S) ? 0 : r;
    }
};

// ------------------------------------------------------------------ received-workers pass
// sel[0..k) = the workers with mask[j] != 0 in increasing order, *kout = k, and
// loss[j] = NaN for the others (their gradients are never formed).  One CTA of
// 1024 threads: a ballot prefix count per warp, then over the warp totals.
__global__ void __launch_bounds__(1024) compact_received_kernel(const uint8_t* __restrict__ mask, int n,
                                                                int32_t* __restrict__ sel, int* __restrict__ kout,
                                                                float* __restrict__ loss, int* __restrict__ zero,
                                                                int nzero) {
    grid_begin();
    __shared__ int warp_tot[32];
    const int j = threadIdx.x, lane = j & 31, warp = j >> 5;
    for (int q = j; q < nzero; q += blockDim.x) zero[q] = 0;
    const bool on = j < n && mask[j] != 0;
    const unsigned bal = __ballot_sync(0xffffffffu, on);
    if (lane == 0) warp_tot[warp] = __popc(bal);
    __syncthreads();
    int base = 0;
    for (int q = 0; q < warp; ++q) base += warp_tot[q];
    if (on) sel[base + __popc(bal & ((1u << lane) - 1u))] = j;
    else if (j < n) loss[j] = NAN;
    if (j == 0) {
        int k = 0;
        for (int q = 0; q < 32; ++q) k += warp_tot[q];
        *kout = k;
    }
}

// Bias part of Eqs. (3)-(4), g[o] = (1/k) sum_{r < k B} dZ[r, o], for every layer,
// in two launches (bias_rows_kernel, mean_update_kernel).  The layers' blocks sit side by
// side in x; a block finds its layer in the prefix table cb0 (blocks of 256 columns).
struct BiasLayers {
    int L;
    const __nv_bfloat16* dz[DBW_LMAX];   // dZ_l [M, ldz]
    int64_t ldz;
    int out[DBW_LMAX];
    int cb0[DBW_LMAX + 1];               // first column block of layer l; cb0[L] = all blocks
    float* part[DBW_LMAX];               // [chunks, out_l] column sums per 256-row chunk
    float* wb[DBW_LMAX];                 // b_l inside w
    float* gb[DBW_LMAX];                 // b_l inside g_t (nullable)
    double* pieces[DBW_LMAX];            // [column blocks of layer l]: pieces of ||g_t(b_l)||^2
};

__device__ __forceinline__ int bias_layer(const BiasLayers& a, int blk) {
    int l = 0;
    while (l + 1 < a.L && blk >= a.cb0[l + 1]) ++l;
    return l;
}

// bias_rows_kernel: one CTA per (layer, 256 columns, 256-row chunk); thread (warp y,
// lane) sums 8 columns (16-byte loads) over rows y, y + 8, ... of the chunk, and the 8
// warps' sums are added in warp order into part[chunk][o].  Chunks past k B write
// nothing.
__global__ void __launch_bounds__(256) bias_rows_kernel(BiasLayers a, int B, const int* __restrict__ kdev) {
    grid_begin();
    __shared__ float red[8][256];
    const int k = *kdev;
    const int rows = k > 0 ? k * B : 0;
    const int r0 = blockIdx.y * 256;
    if (r0 >= rows) return;
    const int l = bias_layer(a, blockIdx.x);
    const int cb = blockIdx.x - a.cb0[l], out = a.out[l];
    const __nv_bfloat16* dZ = a.dz[l];
    const int64_t ldz = a.ldz;
    const int lane = threadIdx.x & 31, y = threadIdx.x >> 5;
    const int c = cb * 256 + 8 * lane;
    float acc[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    const int rend = r0 + 256 < rows ? r0 + 256 : rows;
    if (c < out) {   // rows are ldz (a multiple of 8) long: columns past out are read and dropped
#pragma unroll 8
        for (int r = r0 + y; r < rend; r += 8) {
            const uint4 raw = *reinterpret_cast<const uint4*>(dZ + static_cast<int64_t>(r) * ldz + c);
            const __nv_bfloat16* h = reinterpret_cast<const __nv_bfloat16*>(&raw);
#pragma unroll
            for (int j = 0; j < 8; ++j) acc[j] += __bfloat162float(h[j]);
        }
    }
#pragma unroll
    for (int j = 0; j < 8; ++j) red[y][8 * lane + j] = acc[j];
    __syncthreads();
    const int o = cb * 256 + threadIdx.x;
    if (o < out) {
        float t = 0.f;
        for (int q = 0; q < 8; ++q) t += red[q][threadIdx.x];
        a.part[l][static_cast<int64_t>(blockIdx.y) * out + o] = t;
    }
}

// The tiles of the mean-gradient GEMMs whose K was split (their partial sums are in part):
// layer l's matrix is out x in, ``plan`` its {split tiles, ranges, first split tile}.
struct SplitLayers {
    int out[DBW_LMAX], in[DBW_LMAX];
    const int* plan[DBW_LMAX];
    const float* part[DBW_LMAX];
    float* w[DBW_LMAX];        // W_l inside w
    float* g[DBW_LMAX];        // W_l inside g_t (nullable)
    double* pieces[DBW_LMAX];
};

// One CTA per (layer, 256 columns): g[o] = (1/k) sum of the chunks' sums (chunk order),
// wb[o] -= lr g, gb[o] = g (nullable); the CTA's sum of g^2 (fp64, fixed tree) into
// pieces[column block].
__device__ __forceinline__ void bias_mean_update(const BiasLayers& a, int B, int k, float lr, double* red) {
    const int chunks = k > 0 ? (k * B + 255) / 256 : 0;
    const int l = bias_layer(a, blockIdx.x);
    const int cb = blockIdx.x - a.cb0[l], out = a.out[l];
    const int o = cb * 256 + threadIdx.x;
    double sq = 0.0;
    if (o < out && k > 0) {
        float t = 0.f;
#pragma unroll 16
        for (int q = 0; q < chunks; ++q) t += a.part[l][static_cast<int64_t>(q) * out + o];
        const float g = t * (1.0f / static_cast<float>(k));
        a.wb[l][o] = fmaf(-lr, g, a.wb[l][o]);
        if (a.gb[l]) a.gb[l][o] = g;
        sq = static_cast<double>(g) * g;
    }
    for (int off = 16; off > 0; off >>= 1) sq += __shfl_xor_sync(0xffffffffu, sq, off);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = sq;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int w = 0; w < 8; ++w) t += red[w];
        a.pieces[l][cb] = t;
    }
}

// One block (32 rows x 128 columns) of a split tile: the ranges' partial sums in range order,
// then the GEMM epilogue's g = sum / k, W -= lr g, gbar = g and the sum of g^2.  The partial
// sums hold a row per lane; the step runs along rows, through shared memory.
__device__ __forceinline__ void finish_block(const SplitLayers& s, int l, int item, int k, float lr,
                                             float (*tile)[132], double* red) {
    const int cut = s.plan[l][0], split = s.plan[l][1], whole = s.plan[l][2];
    const int M = s.out[l], N = s.in[l], nt_n = (N + 255) / 256;
    const int j = item >> 4, rank = (item >> 3) & 1, ew = item & 7;
    const int t = whole + j, msub = t / nt_n * 2 + rank, nt = t % nt_n;
    const int q = (ew + 2) & 3, h = ew >> 2;
    const int row0 = msub * 128 + 32 * q, col0 = nt * 256 + 128 * h;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    double sq = 0.0;
    if (row0 < M && col0 < N) {   // the same for the whole block
        const float4* src = reinterpret_cast<const float4*>(s.part[l]) + static_cast<int64_t>(item) * (kTcPartFloats / 4) +
                            warp * 32 + lane;
        const int64_t step = static_cast<int64_t>(cut) * 16 * (kTcPartFloats / 4);
        float4 v[4];
#pragma unroll
        for (int c = 0; c < 4; ++c) v[c] = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 2
        for (int r = 0; r < split; ++r) {
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                if (col0 + 32 * c >= N) continue;
                const float4 x = __ldcg(src + r * step + c * 256);
                v[c].x += x.x;
                v[c].y += x.y;
                v[c].z += x.z;
                v[c].w += x.w;
            }
        }
#pragma unroll
        for (int c = 0; c < 4; ++c) *reinterpret_cast<float4*>(&tile[lane][32 * c + 4 * warp]) = v[c];
        __syncthreads();
        const float inv_k = 1.0f / static_cast<float>(k);
        float* wl = s.w[l];
        float* gl = s.g[l];
        const bool vec = ((reinterpret_cast<uintptr_t>(wl) | reinterpret_cast<uintptr_t>(gl)) & 15u) == 0 && N % 4 == 0;
        const int col = col0 + 4 * lane;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int r = warp + 8 * i, row = row0 + r;
            if (row >= M || col >= N) continue;
            const float4 x = *reinterpret_cast<const float4*>(&tile[r][4 * lane]);
            const float g[4] = {x.x * inv_k, x.y * inv_k, x.z * inv_k, x.w * inv_k};
            const int64_t at = static_cast<int64_t>(row) * N + col;
            if (vec) {
                float4 w = *reinterpret_cast<const float4*>(wl + at);
                w.x = fmaf(-lr, g[0], w.x);
                w.y = fmaf(-lr, g[1], w.y);
                w.z = fmaf(-lr, g[2], w.z);
                w.w = fmaf(-lr, g[3], w.w);
                *reinterpret_cast<float4*>(wl + at) = w;
                if (gl) *reinterpret_cast<float4*>(gl + at) = make_float4(g[0], g[1], g[2], g[3]);
                sq += g[0] * g[0] + g[1] * g[1] + g[2] * g[2] + g[3] * g[3];
            } else {
                for (int e = 0; e < 4 && col + e < N; ++e) {
                    wl[at + e] = fmaf(-lr, g[e], wl[at + e]);
                    if (gl) gl[at + e] = g[e];
                    sq += g[e] * g[e];
                }
            }
        }
    }
    for (int off = 16; off > 0; off >>= 1) sq += __shfl_xor_sync(0xffffffffu, sq, off);
    if (lane == 0) red[warp] = sq;
    __syncthreads();
    if (threadIdx.x == 0 && msub < (M + 127) / 128) {
        double t8 = 0.0;
        for (int w = 0; w < 8; ++w) t8 += red[w];
        s.pieces[l][(static_cast<int64_t>(msub) * nt_n + nt) * 8 + h * 4 + q] = t8;
    }
    __syncthreads();   // tile and red are free again
}

// The bias part of g_t and its step (the first cb0[L] CTAs), and the split tiles of the
// weight part (the others, a block at a time).
__global__ void __launch_bounds__(256) mean_update_kernel(BiasLayers a, SplitLayers s, int B,
                                                          const int* __restrict__ kdev, float lr) {
    grid_begin();
    __shared__ __align__(16) float tile[32][132];
    __shared__ double red[8];
    const int k = *kdev, nb = a.cb0[a.L];
    if (static_cast<int>(blockIdx.x) < nb) {
        bias_mean_update(a, B, k, lr, red);
        return;
    }
    const int step = gridDim.x - nb;
    int item = blockIdx.x - nb;   // counted through the layers
    for (int l = 0; l < a.L; ++l) {
        const int items = s.plan[l][0] * 16;
        for (; item < items; item += step) finish_block(s, l, item, k, lr, tile, red);
        item -= items;
    }
}

struct FinishArgs {
    int L, n, B, CT;
    const double* pw[DBW_LMAX];   // tile pieces of ||g_t(W_l)||^2
    int64_t npw[DBW_LMAX];
    const double* pb[DBW_LMAX];   // CTA pieces of ||g_t(b_l)||^2
    int npb[DBW_LMAX];
    const double* pg[DBW_LMAX];   // Gram pieces, [(row group) * CT + ct]
};

// Writes the partials buffer dbw_grad_stats reads (one block per quantity):
//   vals[j] = ||g_j||^2 for received j (sum over layers and the worker's Gram pieces),
//             0 for the others;
//   vals[n + 1] = ||g_t||^2 (all W and b pieces);
//   vals[n] = sum_j ||g_j||^2 - k ||g_t||^2, the deviation sum of Eq. (10) by the
//             identity sum_j ||g_j - g_t||^2 = sum_j ||g_j||^2 - k ||g_t||^2 (fp64).  Where the
//             workers' gradients are nearly equal (U(0,1) features) the two cancel, and what
//             rounding leaves in ||g_t||^2 shows k-fold: relative error 2.1e-4 at 3072-1024-1024-10,
//             k = 96 (24 inputs; 2.6e-4 with the mean gradient's K in one piece).
// Every sum runs in a fixed order (strided per thread, then a fixed tree).  1024
// threads: the ~12k pieces of the 4096-wide workload are ~12 loads per thread.
constexpr int kFinishThreads = 1024;

__global__ void __launch_bounds__(kFinishThreads) finish_received_kernel(FinishArgs a, const int32_t* __restrict__ sel,
                                                                         const int* __restrict__ kdev,
                                                                         double* __restrict__ partials) {
    grid_begin();
    __shared__ double red[2][32];
    const int t = threadIdx.x, n = a.n, lane = t & 31, warp = t >> 5;
    const int k = *kdev;
    int64_t* hdr = reinterpret_cast<int64_t*>(partials);
    double* vals = partials + kPartialsHeader + (n + 2);
    if (t == 0) {
        hdr[0] = kPartialsMagic;
        hdr[1] = 1;
        hdr[2] = n;
        hdr[3] = 0;
    }
    for (int j = t; j < n; j += kFinishThreads) vals[j] = 0.0;
    double g2 = 0.0, rs = 0.0;
    for (int l = 0; l < a.L; ++l) {
#pragma unroll 8
        for (int64_t i = t; i < a.npw[l]; i += kFinishThreads) g2 += a.pw[l][i];
        for (int i = t; i < a.npb[l]; i += kFinishThreads) g2 += a.pb[l][i];
    }
    __syncthreads();   // zeros above land before the received rows below
    const int per = a.B / 32 * a.CT;   // pieces of a worker and layer: 32-row groups x column tiles
    for (int s = t; s < k; s += kFinishThreads) {
        double v = 0.0;
        for (int l = 0; l < a.L; ++l) {
            const double* pg = a.pg[l] + static_cast<int64_t>(s) * per;
#pragma unroll 8
            for (int i = 0; i < per; ++i) v += pg[i];
        }
        vals[sel[s]] = v;
        rs += v;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        g2 += __shfl_xor_sync(0xffffffffu, g2, o);
        rs += __shfl_xor_sync(0xffffffffu, rs, o);
    }
    if (lane == 0) {
        red[0][warp] = g2;
        red[1][warp] = rs;
    }
    __syncthreads();
    if (t >= 32) return;
    g2 = red[0][lane];
    rs = red[1][lane];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        g2 += __shfl_xor_sync(0xffffffffu, g2, o);
        rs += __shfl_xor_sync(0xffffffffu, rs, o);
    }
    if (t == 0) {
        if (k > 0) {
            vals[n + 1] = g2;
            vals[n] = rs - static_cast<double>(k) * g2;
        } else {
            vals[n + 1] = NAN;
            vals[n] = NAN;
        }
    }
}

}  // namespace

// CTAs of a warp-per-row kernel over ``rows`` rows (8 warps each, at most 8 per SM).
static int row_ctas(int64_t rows) {
    const int64_t want = (rows + 7) / 8, most = 8 * sm_count();
    return static_cast<int>(want < most ? want : most);
}

// bf16 W_l of every layer (one launch).
static void launch_weight_casts(const TcPlan& P, const float* w, char* ws, cudaStream_t st) {
    const GradsPlan& g = P.g;
    WeightCasts a{};
    a.L = g.L;
    a.r0[0] = 0;
    for (int l = 0; l < g.L; ++l) {
        a.w[l] = w + g.offW[l];
        a.fin[l] = g.widths[l];
        a.r0[l + 1] = a.r0[l] + g.widths[l + 1];
        a.vec[l] = aligned16(a.w[l]) && g.widths[l] % 4 == 0;
        a.wb[l] = reinterpret_cast<__nv_bfloat16*>(ws + P.off_wb[l]);
        a.ldw[l] = P.ldw[l];
    }
    launch(cast_weights_kernel, row_ctas(a.r0[g.L]), 256, 0, st, a);
}

bool make_tc_plan(int L, const int32_t* widths, int n, int B, TcPlan* P) {
    GradsPlan g;
    if (!make_grads_plan(L, widths, n, B, DBW_PREC_BF16, &g)) return false;
    P->g = g;
    const int64_t M = static_cast<int64_t>(n) * B;
    int maxw = 0;   // of the layers dZ is formed for
    for (int l = 1; l <= L; ++l) maxw = widths[l] > maxw ? widths[l] : maxw;
    size_t cur = 0;
    auto take = [&](size_t bytes) {
        const size_t at = cur;
        cur += (bytes + 255) / 256 * 256;
        return at;
    };
    P->off_status = take(256);
    P->off_cnt = take(static_cast<size_t>(n) * 4);
    for (int l = 0; l < L; ++l) {
        P->ldw[l] = rup(widths[l], 8);
        P->off_wb[l] = take(static_cast<size_t>(widths[l + 1]) * P->ldw[l] * 2);
    }
    for (int l = 0; l < L; ++l) {   // act[0] = X
        P->ldact[l] = rup(widths[l], 8);
        P->off_act[l] = take(static_cast<size_t>(M) * P->ldact[l] * 2);
    }
    P->ldlog = rup(widths[L], 4);
    P->off_logits = take(static_cast<size_t>(M) * P->ldlog * 4);
    P->off_sloss = take(static_cast<size_t>(M) * 4);
    P->ldz = rup(maxw, 8);
    P->off_dz[0] = take(static_cast<size_t>(M) * P->ldz * 2);
    P->off_dz[1] = take(static_cast<size_t>(M) * P->ldz * 2);
    P->ws_bytes = cur;
    return true;
}

int worker_grads_tc(const TcPlan& P, const float* w, const float* pool, int64_t S, const int32_t* labels,
                    const int32_t* idx, float* G, int64_t ld, float* loss, char* ws, cudaStream_t st) {
    const GradsPlan& g = P.g;
    const int L = g.L, M = g.M, B = g.B, n = g.n;
    int* status = reinterpret_cast<int*>(ws + P.off_status);
    auto bf = [&](size_t off) { return reinterpret_cast<__nv_bfloat16*>(ws + off); };
    int* cnt = reinterpret_cast<int*>(ws + P.off_cnt);
    cudaError_t e = cudaMemsetAsync(status, 0, P.off_cnt - P.off_status + n * sizeof(int), st);   // and the counters
    if (e != cudaSuccess) return fail(DBW_ECUDA, "dbw_worker_grads: %s", cudaGetErrorString(e));

    launch_weight_casts(P, w, ws, st);
    launch(cast_rows_kernel<GatherRows>, row_ctas(M), 256, 0, st, pool, g.widths[0], M, g.widths[0], GatherRows{idx, S},
                                                  bf(P.off_act[0]), P.ldact[0]);
    e = cudaGetLastError();
    if (e != cudaSuccess) return fail(DBW_ECUDA, "dbw_worker_grads: %s", cudaGetErrorString(e));

    // forward
    float* logits = reinterpret_cast<float*>(ws + P.off_logits);
    for (int l = 0; l < L; ++l) {
        const TcOperands fo{bf(P.off_act[l]), P.ldact[l], bf(P.off_wb[l]), P.ldw[l], M, g.widths[l + 1], g.widths[l]};
        TcEpi ep{};
        ep.bias = w + g.offb[l];
        int rc;
        if (l < L - 1) {
            ep.out = bf(P.off_act[l + 1]);
            ep.ldo = P.ldact[l + 1];
            rc = tc_gemm(TC_HIDDEN, fo, ep, status, st);
        } else {
            ep.outF = logits;
            ep.ldF = P.ldlog;
            rc = tc_gemm(TC_LOGITS, fo, ep, status, st);
        }
        if (rc) return rc;
    }
    // loss and dZ_L
    const int C = g.widths[L];
    float* sloss = reinterpret_cast<float*>(ws + P.off_sloss);
    int cur = 0;
    e = launch_softmax(logits, P.ldlog, C, n, B, idx, S, labels, sloss, bf(P.off_dz[0]), P.ldz, loss, cnt, st);
    if (e != cudaSuccess) return fail(DBW_ECUDA, "dbw_worker_grads: %s", cudaGetErrorString(e));

    // backward
    for (int l = L - 1; l >= 0; --l) {
        const int fin = g.widths[l], fout = g.widths[l + 1];
        TcEpi ep{};
        ep.G = G;
        ep.ldG = ld;
        ep.off = g.offW[l];
        ep.ldrow = fin;
        int rc = tc_dw({bf(P.off_dz[cur]), P.ldz, bf(P.off_act[l]), P.ldact[l], fout, fin, B}, n, ep, status, st);
        if (rc) return rc;
        e = launch_bias_grad(bf(P.off_dz[cur]), P.ldz, fout, n, B, G, ld, g.offb[l], st);
        if (e != cudaSuccess) return fail(DBW_ECUDA, "dbw_worker_grads: %s", cudaGetErrorString(e));
        if (l > 0) {
            TcEpi ex{};
            ex.act = bf(P.off_act[l]);
            ex.ldact = P.ldact[l];
            ex.out = bf(P.off_dz[cur ^ 1]);
            ex.ldo = P.ldz;
            rc = tc_gemm(TC_DX, {bf(P.off_dz[cur]), P.ldz, bf(P.off_wb[l]), P.ldw[l], M, fin, fout}, ex, status, st);
            if (rc) return rc;
            cur ^= 1;
        }
    }
    return DBW_OK;
}

// ------------------------------------------------------------------ received-workers pass
// Eqs. (2)-(4) and the statistics of Sect. 3.1 for the k received workers only,
// without the [n, d] gradient matrix: the rows of the received workers are
// stacked (slot s = s-th received worker), the forward and input-gradient GEMMs
// run over those k B rows, the weight part of g_t is one GEMM with K = k B whose
// epilogue applies the SGD step (TC_GBAR), the bias part is a column sum, and the
// per-worker squared norms come from B x B Gram matrices (tc_gram).  The number
// of received workers k is read on the device from ``mask``.

// Whole 32-sample blocks always.  Another B was computed on FFMA tiles, whose sums round in
// another order.  Neither form is the more exact: over 100 random models (B = 16, 50, 100, 200 and
// 500, one to four layers, two inputs each) the error of G against 64 bits here is 0.9994 to 1.003 of
// that on FFMA in each of the 20 classes, 1.000 +- 0.0003 over all.  But a bf16 rounding that falls
// the other way can move a pre-activation across the ReLU's zero, which adds or drops one sample in
// an entry of G: the fewer samples and the more layers, the larger the difference between the two.
// Against the bound of 0.9 of an entry's scale (the rms of G or the entry), 14 random models each:
// with 16 samples up to 1.5, with 50 0.86, with 100 0.71, with 200 and 500 0.49; iterations of four
// layers and more that receive one or two workers pass the bound's 2-norm part (2e-2) at any B (up
// to 3.6e-2), of up to three layers they stay at 8.5e-3.  The line keeps what a call of such a size
// returns within that bound of what it returned before; it is no limit of the kernels, and costs
// time: 16 workers of 500 samples, 3072-1024-1024-10, take 5,440 us on FFMA, 288 here.
bool tc_eligible(int prec, int L, int B) { return prec == DBW_PREC_BF16 && (B % 32 == 0 || (B >= 96 && L <= 3)); }

bool rx_eligible(int prec, int B) {
    return prec == DBW_PREC_BF16 && B % 32 == 0 && (128 % B == 0 || B % 128 == 0);
}

bool make_rx_plan(int L, const int32_t* widths, int n, int B, RxPlan* P) {
    if (!make_tc_plan(L, widths, n, B, &P->t)) return false;
    const GradsPlan& g = P->t.g;
    P->CT = B > 128 ? B / 128 : 1;
    size_t cur = P->t.ws_bytes;
    auto take = [&](size_t bytes) {
        const size_t at = cur;
        cur += (bytes + 255) / 256 * 256;
        return at;
    };
    P->off_sel = take(static_cast<size_t>(n) * 4);
    P->off_k = take(4);
    for (int l = 0; l < L; ++l)   // bias column sums per 256-row chunk, per layer
        P->off_bpart[l] = take(static_cast<size_t>((g.M + 255) / 256) * g.widths[l + 1] * 4);
    // dZ_l of every layer stays until the bias sums and the Gram norms of all layers run
    // after the backward pass: the two ping-pong buffers hold the last two layers'
    for (int l = 0; l < L; ++l) {
        const int back = L - 1 - l;
        P->off_dzl[l] = back < 2 ? P->t.off_dz[back] : take(static_cast<size_t>(g.M) * P->t.ldz * 2);
    }
    for (int l = 0; l < L; ++l) {
        const int fin = g.widths[l], fout = g.widths[l + 1];
        P->npw[l] = static_cast<int64_t>((fout + 127) / 128) * ((fin + 255) / 256) * 8;
        P->off_pw[l] = take(static_cast<size_t>(P->npw[l]) * 8);
        P->npb[l] = (fout + 255) / 256;
        P->off_pb[l] = take(static_cast<size_t>(P->npb[l]) * 8);
        P->off_pg[l] = take(static_cast<size_t>(g.M / 32) * P->CT * 8);
    }
    P->off_gpart = take(tc_gram_partial_floats(g.M, B, L) * 4);
    P->ngcnt = static_cast<int>(tc_gram_items(g.M, B, L));
    P->off_gcnt = take(static_cast<size_t>(P->ngcnt) * 4);
    P->off_split = take(static_cast<size_t>(L) * 16);
    for (int l = 0; l < L; ++l) P->off_part[l] = take(tc_split_floats(g.widths[l + 1], g.widths[l]) * 4);
    P->ws_bytes = cur;
    return true;
}

int received_grads_tc(const RxPlan& P, float* w, const float* pool, int64_t S, const int32_t* labels,
                      const int32_t* idx, const uint8_t* mask, float lr, float* gbar, float* loss, double* partials,
                      char* ws, cudaStream_t st) {
    const TcPlan& T = P.t;
    const GradsPlan& g = T.g;
    const int L = g.L, M = g.M, B = g.B, n = g.n;
    int* status = reinterpret_cast<int*>(ws + T.off_status);
    int32_t* sel = reinterpret_cast<int32_t*>(ws + P.off_sel);
    int* kdev = reinterpret_cast<int*>(ws + P.off_k);
    auto bf = [&](size_t off) { return reinterpret_cast<__nv_bfloat16*>(ws + off); };
    auto f64 = [&](size_t off) { return reinterpret_cast<double*>(ws + off); };
    const char* what = "dbw_received_grads_update";
    int* cnt = reinterpret_cast<int*>(ws + T.off_cnt);
    cudaError_t e = cudaMemsetAsync(status, 0, T.off_cnt - T.off_status + n * sizeof(int), st);   // and the counters
    if (e != cudaSuccess) return fail(DBW_ECUDA, "%s: %s", what, cudaGetErrorString(e));

    int* gcnt = reinterpret_cast<int*>(ws + P.off_gcnt);
    float* gpart = reinterpret_cast<float*>(ws + P.off_gpart);
    launch(compact_received_kernel, 1, 1024, 0, st, mask, n, sel, kdev, loss, gcnt, P.ngcnt);
    launch_weight_casts(T, w, ws, st);
    launch(cast_rows_kernel<ReceivedRows>, row_ctas(M), 256, 0, st, pool, g.widths[0], M, g.widths[0], ReceivedRows{idx, sel, kdev, B, S},
                                                  bf(T.off_act[0]), T.ldact[0]);
    e = cudaGetLastError();
    if (e != cudaSuccess) return fail(DBW_ECUDA, "%s: %s", what, cudaGetErrorString(e));

    // forward over the live rows
    float* logits = reinterpret_cast<float*>(ws + T.off_logits);
    for (int l = 0; l < L; ++l) {
        const TcOperands fo{bf(T.off_act[l]), T.ldact[l], bf(T.off_wb[l]), T.ldw[l], M, g.widths[l + 1], g.widths[l]};
        TcEpi ep{};
        ep.bias = w + g.offb[l];
        ep.kdev = kdev;
        ep.kmul = B;
        int rc;
        if (l < L - 1) {
            ep.out = bf(T.off_act[l + 1]);
            ep.ldo = T.ldact[l + 1];
            rc = tc_gemm(TC_HIDDEN, fo, ep, status, st);
        } else {
            ep.outF = logits;
            ep.ldF = T.ldlog;
            rc = tc_gemm(TC_LOGITS, fo, ep, status, st);
        }
        if (rc) return rc;
    }
    const int C = g.widths[L];
    float* sloss = reinterpret_cast<float*>(ws + T.off_sloss);
    e = launch_softmax(logits, T.ldlog, C, n, B, idx, S, labels, sloss, bf(P.off_dzl[L - 1]), T.ldz, loss, cnt, st, sel,
                       kdev);
    if (e != cudaSuccess) return fail(DBW_ECUDA, "%s: %s", what, cudaGetErrorString(e));

    // backward: per layer the mean gradient with the SGD step and dZ of the layer below in
    // one launch: both read dZ_l, and dZ of every layer is kept in its own buffer.
    for (int l = L - 1; l >= 0; --l) {
        const int fin = g.widths[l], fout = g.widths[l + 1];
        TcEpi gb{};
        gb.W = w;
        gb.gbar = gbar;
        gb.lr = lr;
        gb.off = g.offW[l];
        gb.ldrow = fin;
        gb.pieces = f64(P.off_pw[l]);
        gb.part = reinterpret_cast<float*>(ws + P.off_part[l]);
        gb.plan = reinterpret_cast<int*>(ws + P.off_split) + 4 * l;
        gb.kdev = kdev;
        gb.kmul = B;
        const TcOperands go{bf(P.off_dzl[l]), T.ldz, bf(T.off_act[l]), T.ldact[l], fout, fin, M};
        int rc;
        if (l > 0) {
            TcEpi ex{};
            ex.act = bf(T.off_act[l]);
            ex.ldact = T.ldact[l];
            ex.out = bf(P.off_dzl[l - 1]);
            ex.ldo = T.ldz;
            ex.kdev = kdev;
            ex.kmul = B;
            const TcOperands xo{bf(P.off_dzl[l]), T.ldz, bf(T.off_wb[l]), T.ldw[l], M, fin, fout};
            rc = tc_gemm_mean_dx(go, gb, xo, ex, status, st);
        } else {
            rc = tc_gemm(TC_GBAR, go, gb, status, st);
        }
        if (rc) return rc;
    }
    // bias part of g_t and its step, every layer in two launches; the second one also finishes
    // the split tiles of the mean-gradient GEMMs
    {
        BiasLayers bl{};
        SplitLayers sl{};
        int most = 0;
        bl.L = L;
        bl.ldz = T.ldz;
        bl.cb0[0] = 0;
        for (int l = 0; l < L; ++l) {
            bl.dz[l] = bf(P.off_dzl[l]);
            bl.out[l] = g.widths[l + 1];
            bl.cb0[l + 1] = bl.cb0[l] + P.npb[l];
            bl.part[l] = reinterpret_cast<float*>(ws + P.off_bpart[l]);
            bl.wb[l] = w + g.offb[l];
            bl.gb[l] = gbar ? gbar + g.offb[l] : nullptr;
            bl.pieces[l] = f64(P.off_pb[l]);
            sl.out[l] = g.widths[l + 1];
            sl.in[l] = g.widths[l];
            sl.plan[l] = reinterpret_cast<const int*>(ws + P.off_split) + 4 * l;
            sl.part[l] = reinterpret_cast<const float*>(ws + P.off_part[l]);
            sl.w[l] = w + g.offW[l];
            sl.g[l] = gbar ? gbar + g.offW[l] : nullptr;
            sl.pieces[l] = f64(P.off_pw[l]);
            most += tc_split_items(g.widths[l + 1], g.widths[l]) * 8;   // a split tile has 2 ranges or more
        }
        launch(bias_rows_kernel, dim3(bl.cb0[L], (M + 255) / 256), 256, 0, st, bl, B, kdev);
        const int ctas = 8 * sm_count();   // all at once: 373 -> 368 us a step over four per SM
        launch(mean_update_kernel, bl.cb0[L] + (most < ctas ? most : ctas), 256, 0, st, bl, sl, B, kdev, lr);
        e = cudaGetLastError();
        if (e != cudaSuccess) return fail(DBW_ECUDA, "%s: %s", what, cudaGetErrorString(e));
    }
    // per-worker norms of every layer in one launch
    {
        const __nv_bfloat16* acts[DBW_LMAX];
        const __nv_bfloat16* dzs[DBW_LMAX];
        int64_t lds[DBW_LMAX];
        int cin[DBW_LMAX], cout[DBW_LMAX];
        double* pg[DBW_LMAX];
        for (int l = 0; l < L; ++l) {
            acts[l] = bf(T.off_act[l]);
            lds[l] = T.ldact[l];
            cin[l] = g.widths[l];
            dzs[l] = bf(P.off_dzl[l]);
            cout[l] = g.widths[l + 1];
            pg[l] = f64(P.off_pg[l]);
        }
        const int rc = tc_gram(L, acts, lds, cin, dzs, T.ldz, cout, M, B, kdev, pg, gpart, gcnt, status, st);
        if (rc) return rc;
    }
    FinishArgs fa{};
    fa.L = L;
    fa.n = n;
    fa.B = B;
    fa.CT = P.CT;
    for (int l = 0; l < L; ++l) {
        fa.pw[l] = f64(P.off_pw[l]);
        fa.npw[l] = P.npw[l];
        fa.pb[l] = f64(P.off_pb[l]);
        fa.npb[l] = P.npb[l];
        fa.pg[l] = f64(P.off_pg[l]);
    }
    launch(finish_received_kernel, 1, kFinishThreads, 0, st, fa, sel, kdev, partials);
    e = cudaGetLastError();
    if (e != cudaSuccess) return fail(DBW_ECUDA, "%s: %s", what, cudaGetErrorString(e));
    return DBW_OK;
}

size_t received_workspace_bytes(int L, const int32_t* widths, int n, int B, int prec) {
    RxPlan P;
    if (!rx_eligible(prec, B) || !make_rx_plan(L, widths, n, B, &P)) return 0;
    return P.ws_bytes;
}

int launch_received_grads(int L, const int32_t* widths, int prec, float* w, int64_t d, const float* pool, int64_t S,
                          const int32_t* labels, const int32_t* idx, int n, int B, const uint8_t* mask, float lr,
                          float* gbar, float* loss, double* partials, void* ws, size_t ws_bytes, cudaStream_t st) {
    const char* what = "dbw_received_grads_update";
    if (!rx_eligible(prec, B))
        return fail(DBW_EUNSUPPORTED, "%s: needs prec = DBW_PREC_BF16, B %% 32 == 0 and B | 128 or 128 | B", what);
    RxPlan P;
    if (!make_rx_plan(L, widths, n, B, &P)) return fail(DBW_EINVAL, "%s: invalid model shape", what);
    if (d != P.t.g.d) return fail(DBW_EINVAL, "%s: d = %lld, the widths give %lld", what, (long long)d,
                                  (long long)P.t.g.d);
    if (ws_bytes < P.ws_bytes) return fail(DBW_EINVAL, "%s: workspace %zu bytes < %zu needed", what, ws_bytes, P.ws_bytes);
    return received_grads_tc(P, w, pool, S, labels, idx, mask, lr, gbar, loss, partials, static_cast<char*>(ws), st);
}

}  // namespace dbw
