// Loss, dZ_L and bias-gradient kernels shared by the fp32 pass (grads.cu) and the bf16
// pass (grads_tc.cu); T is the type of dZ.
#pragma once

#include <cuda_bf16.h>
#include <math.h>

#include "common.cuh"

namespace dbw {
namespace {

template <typename T> __device__ __forceinline__ T from_f(float v);
template <> __device__ __forceinline__ float from_f<float>(float v) { return v; }
template <> __device__ __forceinline__ __nv_bfloat16 from_f<__nv_bfloat16>(float v) { return __float2bfloat16_rn(v); }

// Rows of the stacked buffers that a received-workers pass computes: the k B
// received rows rounded up to the 128-row GEMM tile (all M when kdev is null).
__device__ __forceinline__ int live_rows(const int* kdev, int B, int M) {
    if (!kdev) return M;
    const int k = *kdev;
    const long long r = (static_cast<long long>(k > 0 ? k : 0) * B + 127) / 128 * 128;
    return r < M ? static_cast<int>(r) : M;
}

// ------------------------------------------------------------------ loss
// Per sample: stable log-softmax cross entropy, and dZ = (softmax - onehot) / B.  A
// worker's loss is the mean of its B sample losses.  A sample index outside [0, S) or a
// label outside [0, C) makes the sample's loss and dZ row NaN, and so the worker's loss and
// gradient.
//
// CTA (i, y) takes rows y rows_cta .. of worker i, a warp kRows rows at a time: their
// logits, sample indices and labels are all loaded before the first is reduced, and a lane
// keeps its NJ logits of a row (classes lane, lane + 32, ..) in registers, so that each is
// read once (NJ = 0, C > 1024: three passes over the row).  (One CTA per worker, a row at a
// time per warp, 32 masked exponentials a row: 45 us for 16,384 rows of 10 classes in bf16, 49 for 16 workers of 500
// in fp32; now 9 and 8.)
//
// With ``sel`` (received-workers pass): slot i is worker sel[i] (stacked rows i B .., samples
// idx[sel[i] B + r], loss[sel[i]]); slots i >= k zero their dZ rows up to the live row count.
constexpr int kLossThreads = 256;

// The CTA that finishes a worker last of its ``parts`` (all T threads call it) adds the worker's
// B sample losses in sample order (part of the loss's definition: F^ enters Eq. (12) as a
// difference), from shared memory, into *loss.  *cnt is zero before the worker's first CTA.
template <int T>
__device__ __forceinline__ void finish_worker_loss(const float* __restrict__ sample_loss, int B, int parts,
                                                   int* __restrict__ cnt, float invB, float* __restrict__ loss) {
    __shared__ int last_s;
    __syncthreads();
    if (threadIdx.x == 0) {
        last_s = 1;
        if (parts > 1) {
            __threadfence();
            last_s = atomicAdd(cnt, 1) == parts - 1;
            __threadfence();
        }
    }
    __syncthreads();
    if (!last_s) return;
    constexpr int kStage = 1024;
    __shared__ __align__(16) float ls[kStage];
    float acc = 0.f;
    for (int s0 = 0; s0 < B; s0 += kStage) {
        const int len = B - s0 < kStage ? B - s0 : kStage;
        for (int r = threadIdx.x; r < kStage; r += T)
            if (r < len) ls[r] = __ldcg(sample_loss + s0 + r);
        __syncthreads();
        if (threadIdx.x == 0) {
            int r = 0;
#pragma unroll 4
            for (; r + 4 <= len; r += 4) {
                const float4 v = *reinterpret_cast<const float4*>(ls + r);
                acc += v.x;
                acc += v.y;
                acc += v.z;
                acc += v.w;
            }
            for (; r < len; ++r) acc += ls[r];
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) *loss = acc * invB;
}

template <int NJ>
constexpr int loss_rows() { return NJ == 1 ? 4 : NJ == 4 ? 2 : 1; }   // rows a warp has in flight

template <typename T, int NJ>
__global__ void __launch_bounds__(kLossThreads) softmax_xent_kernel(
    const float* __restrict__ logits, int64_t ldl, int C, int B, int rows_cta, const int32_t* __restrict__ idx,
    int64_t S, const int32_t* __restrict__ labels, float* __restrict__ sample_loss, T* __restrict__ dZ, int64_t ldz,
    float* __restrict__ loss, int* __restrict__ cnt, const int32_t* __restrict__ sel, const int* __restrict__ kdev) {
    grid_begin();
    constexpr int RW = loss_rows<NJ>();
    const int i = blockIdx.x;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = kLossThreads / 32;
    const int64_t row0 = static_cast<int64_t>(i) * B;
    const int rbeg = blockIdx.y * rows_cta, rend = rbeg + rows_cta < B ? rbeg + rows_cta : B;
    int worker = i;
    if (sel) {
        if (i >= *kdev) {
            const int64_t live = live_rows(kdev, B, gridDim.x * B);
            for (int r = rbeg + warp; r < rend && row0 + r < live; r += nw)
                for (int c = lane; c < C; c += 32) dZ[(row0 + r) * ldz + c] = from_f<T>(0.f);
            return;
        }
        worker = sel[i];
    }
    const float invB = 1.0f / static_cast<float>(B);
    for (int r0 = rbeg + warp * RW; r0 < rend; r0 += nw * RW) {
        int ymine = -1;   // lane u: label of row r0 + u
        if (lane < RW && r0 + lane < rend) {
            const int64_t sidx = idx[static_cast<int64_t>(worker) * B + r0 + lane];
            if (sidx >= 0 && sidx < S) ymine = labels[sidx];
        }
        float z[RW][NJ > 0 ? NJ : 1];
        if constexpr (NJ > 0) {
#pragma unroll
            for (int u = 0; u < RW; ++u)
#pragma unroll
                for (int j = 0; j < NJ; ++j) {
                    const int c = lane + 32 * j;
                    z[u][j] = r0 + u < rend && c < C ? logits[(row0 + r0 + u) * ldl + c] : -INFINITY;
                }
        }
#pragma unroll
        for (int u = 0; u < RW; ++u) {
            const int r = r0 + u;
            if (r >= rend) break;
            const int y = __shfl_sync(0xffffffffu, ymine, u);
            const bool bad = (y < 0 || y >= C);
            const float* zr = logits + (row0 + r) * ldl;
            T* dzr = dZ + (row0 + r) * ldz;
            float mx = -INFINITY, se = 0.f, zy;
            if constexpr (NJ > 0) {
#pragma unroll
                for (int j = 0; j < NJ; ++j) mx = fmaxf(mx, z[u][j]);
            } else {
                for (int c = lane; c < C; c += 32) mx = fmaxf(mx, zr[c]);
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
            if constexpr (NJ > 0) {
                zy = 0.f;
#pragma unroll
                for (int j = 0; j < NJ; ++j) {
                    if (lane + 32 * j == y) zy = z[u][j];
                    z[u][j] = lane + 32 * j < C ? expf(z[u][j] - mx) : 0.f;
                    se += z[u][j];
                }
                zy = __shfl_sync(0xffffffffu, zy, y & 31);
            } else {
                for (int c = lane; c < C; c += 32) se += expf(zr[c] - mx);
                zy = bad ? 0.f : zr[y];
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) se += __shfl_xor_sync(0xffffffffu, se, o);
            const float inv_se = 1.0f / se;
            if constexpr (NJ > 0) {
#pragma unroll
                for (int j = 0; j < NJ; ++j) {
                    const int c = lane + 32 * j;
                    float g = z[u][j] * inv_se;
                    if (c == y) g -= 1.0f;
                    if (c < C) dzr[c] = from_f<T>(bad ? NAN : g * invB);
                }
            } else {
                for (int c = lane; c < C; c += 32) {
                    float g = expf(zr[c] - mx) * inv_se;
                    if (c == y) g -= 1.0f;
                    dzr[c] = from_f<T>(bad ? NAN : g * invB);
                }
            }
            if (lane == 0) sample_loss[row0 + r] = bad ? NAN : (mx + logf(se)) - zy;
        }
    }
    finish_worker_loss<kLossThreads>(sample_loss + row0, B, gridDim.y, cnt + i, invB, loss + worker);
}

template <typename T>
cudaError_t launch_softmax(const float* logits, int64_t ldl, int C, int n, int B, const int32_t* idx, int64_t S,
                           const int32_t* labels, float* sample_loss, T* dZ, int64_t ldz, float* loss, int* cnt,
                           cudaStream_t st, const int32_t* sel = nullptr, const int* kdev = nullptr) {
    // two passes of a CTA's warps over their rows in flight, more where the grid's y would overflow
    const int per_pass = kLossThreads / 32 * (C <= 32 ? loss_rows<1>() : C <= 128 ? loss_rows<4>() : 1);
    int rows_cta = 2 * per_pass;
    while ((B + rows_cta - 1) / rows_cta > 65535) rows_cta *= 2;
    const dim3 grid(n, (B + rows_cta - 1) / rows_cta);
    auto kern = C <= 32 ? softmax_xent_kernel<T, 1> : C <= 128 ? softmax_xent_kernel<T, 4>
              : C <= 1024 ? softmax_xent_kernel<T, 32> : softmax_xent_kernel<T, 0>;
    launch(kern, grid, kLossThreads, 0, st, logits, ldl, C, B, rows_cta, idx, S, labels, sample_loss, dZ, ldz, loss, cnt,
                                        sel, kdev);
    return cudaGetLastError();
}

// ------------------------------------------------------------------ bias gradient
// G[i, offb + o] = sum_{r < B} dZ[i B + r, o].  A thread owns V neighbouring columns (one load
// of V elements a row) and every RL-th row, RL = kBiasThreads / CG row lanes beside CG column
// groups; the row lanes' sums are then added in a fixed tree.  (A thread per column over
// all rows, the loads of a row 2 or 4 bytes a lane: 38 us for the three layers of
// 3072-1024-1024-10 at n = B = 128, 60 at 16 workers of 500; now 27 and 25.)
constexpr int kBiasThreads = 256;

template <typename T, int V> struct BiasVec;   // V elements as one load
template <> struct BiasVec<float, 1> { using type = float; };
template <> struct BiasVec<float, 2> { using type = float2; };
template <> struct BiasVec<float, 4> { using type = float4; };
template <> struct BiasVec<__nv_bfloat16, 1> { using type = __nv_bfloat16; };
template <> struct BiasVec<__nv_bfloat16, 8> { using type = uint4; };

__device__ __forceinline__ float bias_to_f(float v) { return v; }
__device__ __forceinline__ float bias_to_f(__nv_bfloat16 v) { return __bfloat162float(v); }

template <typename T, int V>
__global__ void __launch_bounds__(kBiasThreads) bias_grad_kernel(const T* __restrict__ dZ, int64_t ldz, int out, int B,
                                                                 int CG, float* __restrict__ G, int64_t ldG,
                                                                 int64_t offb) {
    grid_begin();
    using Vec = typename BiasVec<T, V>::type;
    __shared__ float red[kBiasThreads * V];
    const int i = blockIdx.y;
    const int cg = threadIdx.x % CG, rl = threadIdx.x / CG, RL = kBiasThreads / CG;
    const int c = (blockIdx.x * CG + cg) * V;
    float acc[V];
#pragma unroll
    for (int v = 0; v < V; ++v) acc[v] = 0.f;
    if (c < out) {   // out is a multiple of V, or the row padding after it is readable (never stored)
        const T* p = dZ + static_cast<int64_t>(i) * B * ldz + c;
#pragma unroll 8
        for (int r = rl; r < B; r += RL) {
            const Vec x = *reinterpret_cast<const Vec*>(p + static_cast<int64_t>(r) * ldz);
            const T* e = reinterpret_cast<const T*>(&x);
#pragma unroll
            for (int v = 0; v < V; ++v) acc[v] += bias_to_f(e[v]);
        }
    }
#pragma unroll
    for (int v = 0; v < V; ++v) red[v * kBiasThreads + threadIdx.x] = acc[v];
    __syncthreads();
    for (int h = RL / 2; h > 0; h >>= 1) {
        if (rl < h) {
#pragma unroll
            for (int v = 0; v < V; ++v)
                red[v * kBiasThreads + threadIdx.x] += red[v * kBiasThreads + threadIdx.x + h * CG];
        }
        __syncthreads();
    }
    // the sums of the block's CG V columns, in column order
    for (int e = threadIdx.x; e < CG * V; e += kBiasThreads) {
        const int o = blockIdx.x * CG * V + e;
        if (o < out) G[static_cast<int64_t>(i) * ldG + offb + o] = red[(e % V) * kBiasThreads + e / V];
    }
}

template <typename T, int V>
cudaError_t launch_bias_v(const T* dZ, int64_t ldz, int out, int n, int B, float* G, int64_t ldG, int64_t offb,
                          cudaStream_t st) {
    // column groups: as many as the columns need, at most a warp's worth, so that a row is
    // read in whole lines and the other threads share the rows; fewer, down to one 128-byte
    // line, while that leaves SMs without a CTA
    int CG = 1;
    while (CG < 32 && CG * V < out) CG *= 2;
    const int line = 128 / (static_cast<int>(sizeof(T)) * V);
    while (CG > line && static_cast<int64_t>((out + CG * V - 1) / (CG * V)) * n < 2 * sm_count()) CG /= 2;
    launch(bias_grad_kernel<T, V>, dim3((out + CG * V - 1) / (CG * V), n), kBiasThreads, 0, st, dZ, ldz, out, B, CG, G, ldG,
                                                                                            offb);
    return cudaGetLastError();
}

// dZ 16-byte aligned.  Wide loads where the rows allow them (the tcgen05 pass pads its bf16 rows
// to 8; the rows of the FFMA pass are as wide as the layer).
inline cudaError_t launch_bias_grad(const float* dZ, int64_t ldz, int out, int n, int B, float* G, int64_t ldG,
                                    int64_t offb, cudaStream_t st) {
    if (ldz % 4 == 0 && out % 4 == 0) return launch_bias_v<float, 4>(dZ, ldz, out, n, B, G, ldG, offb, st);
    if (ldz % 2 == 0 && out % 2 == 0) return launch_bias_v<float, 2>(dZ, ldz, out, n, B, G, ldG, offb, st);
    return launch_bias_v<float, 1>(dZ, ldz, out, n, B, G, ldG, offb, st);
}
inline cudaError_t launch_bias_grad(const __nv_bfloat16* dZ, int64_t ldz, int out, int n, int B, float* G, int64_t ldG,
                                    int64_t offb, cudaStream_t st) {
    if (out >= 8 && ldz % 8 == 0) return launch_bias_v<__nv_bfloat16, 8>(dZ, ldz, out, n, B, G, ldG, offb, st);
    return launch_bias_v<__nv_bfloat16, 1>(dZ, ldz, out, n, B, G, ldG, offb, st);
}

}  // namespace
}  // namespace dbw
