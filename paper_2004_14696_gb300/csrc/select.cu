// Eq. (4): arrival order of the n gradients and the k = n - b the PS keeps.
//
// Worker i's arrival rank is the number of workers j with (T_j, j) < (T_i, i).  A warp
// ranks one worker: each lane compares it with a 1/32 slice of the workers and the counts
// meet in a warp reduction.  Ranks of a strict total order are a permutation, which gives
// order, mask and the order statistics directly, so the warps share nothing and spread
// over the SMs (one CTA whose 8 warps ranked 32 workers each took 8 us at n = 256).
//
// The comparisons run on 64-bit integer keys: a double's bits, with the sign bit
// flipped for non-negative values and all bits flipped for negative ones (-0 is
// first made +0), order exactly as the doubles do and are equal exactly when the
// doubles are.  On this part a dependent fp64 compare costs ~12x an integer one.
#include "common.cuh"

namespace dbw {

namespace {
__device__ __forceinline__ unsigned long long order_key(double t) {
    unsigned long long u = static_cast<unsigned long long>(__double_as_longlong(t));
    if (u == 0x8000000000000000ull) u = 0;   // -0 == +0
    return (u >> 63) ? ~u : (u | 0x8000000000000000ull);
}
}  // namespace

constexpr int kSelectWarps = 8;

// Only a launch of one CTA, which stages every time and reads b before its first store, may have
// times in tsorted's memory or b in k_out's.
__global__ void __launch_bounds__(1024) select_fastest_kernel(
    const double* times, int n, const int32_t* b_ptr,
    int32_t* __restrict__ order, uint8_t* __restrict__ mask, double* tsorted,
    int32_t* k_out) {
    grid_begin();
    __shared__ double ts[DBW_NMAX];
    __shared__ unsigned long long key[DBW_NMAX];
    int b = *b_ptr;
    for (int j = threadIdx.x; j < n; j += blockDim.x) {
        const double t = times[j];
        ts[j] = t;
        key[j] = order_key(t);
    }
    __syncthreads();
    b = b < 0 ? 0 : (b > n - 1 ? n - 1 : b);
    const int k = n - b;
    const int lane = threadIdx.x & 31, warps = blockDim.x >> 5;
    for (int i = blockIdx.x * warps + (threadIdx.x >> 5); i < n; i += gridDim.x * warps) {
        const unsigned long long ki = key[i];
        int rank = 0;
#pragma unroll 4
        for (int j = lane; j < n; j += 32) {
            const unsigned long long kj = key[j];
            rank += (kj < ki) || (kj == ki && j < i);
        }
        rank = __reduce_add_sync(0xffffffffu, rank);
        if (lane == 0) {
            order[rank] = i;
            tsorted[rank] = ts[i];
            mask[i] = rank < k ? 1 : 0;
        }
    }
    if (blockIdx.x == 0 && threadIdx.x == 0 && k_out) *k_out = k;
}

cudaError_t launch_select(const double* times, int n, const int32_t* b, int32_t* order,
                          uint8_t* mask, double* tsorted, int32_t* k_out, cudaStream_t st) {
    if ((times < tsorted + n && tsorted < times + n) || k_out == b)   // over its own inputs: one CTA
        launch(select_fastest_kernel, 1, 1024, 0, st, times, n, b, order, mask, tsorted, k_out);
    else
        launch(select_fastest_kernel, (n + kSelectWarps - 1) / kSelectWarps, 32 * kSelectWarps, 0, st, 
            times, n, b, order, mask, tsorted, k_out);
    return cudaGetLastError();
}

}  // namespace dbw
