// The DBW estimator on the device (Sect. 3): end-of-iteration statistics
// (Eqs. (10)-(12), time bookkeeping of Sect. 3.2) and the choice of k_t
// (Eqs. (13)-(19)).  Everything is fp64 and runs in one CTA.
//
// This file is compiled with -fmad=false: every multiply and add below is a
// separately rounded IEEE operation, performed in the order written, so that a
// state reproduced elsewhere with the same operation order yields the same b_t
// bit for bit.  The window sums and the loss sum are defined as sequential sums; the
// loss sum runs in parallel whenever every order of it is exact (loss_sum below), and
// independent divisions run in different lanes of one warp.  Inputs are first loaded
// into shared memory by all threads, and so are the state's scalar fields (one round
// trip instead of one per field).
#include <math.h>
#include <math_constants.h>
#include <stddef.h>

#include "common.cuh"

namespace dbw {

namespace {

constexpr int kRedThreads = 256;

__device__ __forceinline__ int ring_slot(int cnt_minus_v) { return cnt_minus_v % DBW_DMAX; }

__device__ double window_mean(const double* ring, int cnt, int D) {
    const int m = cnt < D ? cnt : D;
    double acc = 0.0;
    for (int v = 1; v <= m; ++v) acc = acc + ring[ring_slot(cnt - v)];
    return acc / (double)m;
}

// The state's scalar fields (everything before the rings), copied into shared memory by
// the first threads in one round trip; the sequential code then reads the copy and
// writes its results to the state itself.
constexpr int kHeadWords = static_cast<int>(offsetof(dbw_state, ringV) / 8);
static_assert(offsetof(dbw_state, ringV) % 8 == 0, "the state's scalar fields are whole 8-byte words");

__device__ __forceinline__ const dbw_state* stage_head(const dbw_state* st, unsigned long long* head) {
    if (threadIdx.x < kHeadWords) head[threadIdx.x] = reinterpret_cast<const unsigned long long*>(st)[threadIdx.x];
    __syncthreads();
    return reinterpret_cast<const dbw_state*>(head);
}

// Sum of the per-block pieces of one quantity, in a fixed order: thread t adds blocks
// t, t + 256, ... sequentially, then a pairwise tree (t adds t + 128, t + 64, ..., t + 1).
// Valid in thread 0; ``red``: shared, kRedThreads.
__device__ __forceinline__ double tree_sum(double s, double* red) {
    const int t = threadIdx.x;
    red[t] = s;
    __syncthreads();
    if (t < 128) red[t] = red[t] + red[t + 128];
    __syncthreads();
    if (t < 64) red[t] = red[t] + red[t + 64];
    __syncthreads();
    if (t < 32) {
        s = red[t] + red[t + 32];
#pragma unroll
        for (int h = 16; h > 0; h >>= 1) s = s + __shfl_down_sync(0xffffffffu, s, h);
    }
    return s;
}
__device__ __forceinline__ double strided_sum(const double* __restrict__ vals, int blocks) {
    double s = 0.0;
    for (int i = threadIdx.x; i < blocks; i += kRedThreads) s = s + vals[i];
    return s;
}

// Sum of the received workers' losses in increasing worker order, in fp64 (in thread 0).
// Floats whose exponent fields span at most 19 are integer multiples, below 2^43, of one
// power of two, so every partial sum of up to 1024 of them fits fp64's 53 bits: no
// addition rounds, whatever the order, and the parallel sum is the sequential one bit for
// bit.  Other inputs (a wider span, infinities, NaN) take the sequential loop in thread 0.
// That loop alone was 256 dependent fp64 additions, about 10 of the 23 us the statistics
// took at n = 256.
__device__ double loss_sum(const float* loss_s, const uint8_t* mask_s, int n, double* red, unsigned* span) {
    const int t = threadIdx.x;
    unsigned lo = 255u, hi = 0u;
    double s = 0.0;
    for (int j = t; j < n; j += kRedThreads) {
        if (!mask_s[j]) continue;
        const unsigned u = __float_as_uint(loss_s[j]) & 0x7fffffffu;
        if (u) {
            const unsigned e = u >> 23 ? u >> 23 : 1u;   // subnormals count in units of exponent field 1
            lo = e < lo ? e : lo;
            hi = e > hi ? e : hi;
        }
        s = s + (double)loss_s[j];
    }
    lo = __reduce_min_sync(0xffffffffu, lo);
    hi = __reduce_max_sync(0xffffffffu, hi);
    if ((t & 31) == 0) {
        atomicMin(span, lo);
        atomicMax(span + 1, hi);
    }
    s = tree_sum(s, red);   // (its barriers order the span)
    if (t == 0 && (span[1] == 255u || (span[1] > span[0] && span[1] - span[0] > 19u))) {
        s = 0.0;
        for (int j = 0; j < n; ++j)
            if (mask_s[j]) s = s + (double)loss_s[j];
    }
    return s;
}

// The statistics of an iteration in one launch: block 0 reduces the two sums of Eqs.
// (10)-(11) it needs, forms the statistics and records them; block 1 + j reduces row j's
// squared norm.  No block waits for another.  (As a reduction launch and then a one-CTA
// launch whose thread 0 counted the mask and summed the losses alone this took 4 + 23 us
// at n = 256, 3 + 6 us at n = 16.)
__global__ void __launch_bounds__(kRedThreads) grad_stats_kernel(
    double* __restrict__ partials, int n, const uint8_t* __restrict__ mask,
    const float* __restrict__ loss, const double* __restrict__ tsorted, double lr,
    dbw_state* __restrict__ st, double* __restrict__ stats_out, double* __restrict__ row_sqnorm) {
    grid_begin();
    __shared__ double red[kRedThreads];
    const int tid = threadIdx.x;
    const int64_t* hdr = reinterpret_cast<const int64_t*>(partials);
    double* sums = partials + kPartialsHeader;
    const double* vals = sums + (n + 2);
    // not written by dbw_aggregate_update for this n: poison instead of reading
    const bool valid = hdr[0] == kPartialsMagic && hdr[2] == n && hdr[1] >= 1 && hdr[1] <= (1 << 20);
    const int blocks = valid ? (int)hdr[1] : 0;
    if (blockIdx.x > 0) {
        const int j = blockIdx.x - 1;
        const bool state_ok = st->n == n;
        int any = 0;
        for (int i = tid; i < n; i += kRedThreads) any |= mask[i];
        const double part = strided_sum(vals + (int64_t)j * blocks, blocks);
        any = __syncthreads_or(any);
        const double total = tree_sum(part, red);
        if (tid == 0) {
            const double v = valid ? total : CUDART_NAN;
            sums[j] = v;
            // the partials header says whether the rows the mask left out were read too
            const bool all_rows = (hdr[3] & DBW_ALL_ROW_NORMS) != 0;
            if (row_sqnorm && any && state_ok) row_sqnorm[j] = (mask[j] || all_rows) ? v : CUDART_NAN;
        }
        return;
    }
    __shared__ uint8_t mask_s[DBW_NMAX];
    __shared__ float loss_s[DBW_NMAX];
    __shared__ unsigned long long head_s[kHeadWords];
    __shared__ double red2[kRedThreads], red3[kRedThreads];
    __shared__ unsigned span[2];
    int mine = 0;
    for (int j = tid; j < n; j += kRedThreads) {   // n <= DBW_NMAX: checked by the caller
        mask_s[j] = mask[j] ? 1 : 0;
        loss_s[j] = loss[j];
        mine += mask_s[j];
    }
    if (tid == 0) {
        span[0] = 255u;
        span[1] = 0u;
    }
    // a block of the aggregation whose wait ran out marks its pieces: w has not taken its whole step
    int lost = 0;
    double ss_part = 0.0;   // strided_sum's order
    for (int i = tid; i < blocks; i += kRedThreads) {
        const double piece = vals[(int64_t)n * blocks + i];
        lost |= __double_as_longlong(piece) == kPieceTimedOut;
        ss_part = ss_part + piece;
    }
    const double g2_part = strided_sum(vals + (int64_t)(n + 1) * blocks, blocks);
    const dbw_state* sh = stage_head(st, head_s);   // (its barrier also orders mask_s, loss_s, span)
    __shared__ int k_s, lost_s;
    if (tid == 0) k_s = lost_s = 0;
    const double SS0 = tree_sum(ss_part, red);      // (its barriers order k_s = 0)
    mine = __reduce_add_sync(0xffffffffu, mine);
    if ((tid & 31) == 0) atomicAdd(&k_s, mine);
    if (lost) lost_s = 1;
    const double g20 = tree_sum(g2_part, red2);     // (its barriers complete k_s)
    const double SS = valid ? SS0 : CUDART_NAN, g2 = valid ? g20 : CUDART_NAN;
    if (tid == 0) {
        sums[n] = SS;
        sums[n + 1] = g2;
    }
    const int k = k_s;
    if (k == 0 || sh->n != n || lost_s) {
        if (tid == 0)
            st->flags = sh->flags | (k == 0 ? DBW_FLAG_EMPTY_MASK : 0) | (sh->n != n ? DBW_FLAG_BAD_STATE : 0) |
                        (lost_s ? DBW_FLAG_WAIT_TIMEOUT : 0);
        return;
    }
    // Sect. 3.2: every arrival is observed, S[r] accumulates the r-th order statistic
    for (int r = tid; r < n; r += kRedThreads) st->S[r] = st->S[r] + tsorted[r];
    const double acc = loss_sum(loss_s, mask_s, n, red3, span);
    if (tid < 32) {
        // the divisions, independent ones in different lanes: lane 0 V^+ of Eq. (10), lane 1
        // F^_t, lane 2 the V / k of Eq. (12); then lane 0 the V^+ / k of Eq. (11), lane 1 Eq. (12)
        const int lane = tid;
        const double SSw = __shfl_sync(0xffffffffu, SS, 0), accw = __shfl_sync(0xffffffffu, acc, 0);
        const double g2w = __shfl_sync(0xffffffffu, g2, 0);
        const double num1 = lane == 0 ? SSw : lane == 1 ? accw : sh->V_last;
        const double den1 = lane == 0 ? (double)(k - 1) : lane == 1 ? (double)k : (double)sh->k_last;
        const double d1 = num1 / den1;
        double V = __shfl_sync(0xffffffffu, d1, 0);
        const double F = __shfl_sync(0xffffffffu, d1, 1);
        const double Vk_last = __shfl_sync(0xffffffffu, d1, 2);
        const double num = 2.0 * ((lr * sh->N_last) - (sh->F_last - F));
        const double den = (lr * lr) * (sh->N_last + Vk_last);
        const double d2 = (lane == 0 ? V : num) / (lane == 0 ? (double)k : den);
        const double Vk = __shfl_sync(0xffffffffu, d2, 0);
        const double L12 = __shfl_sync(0xffffffffu, d2, 1);
        if (lane == 0) {
            double N = CUDART_NAN, L = CUDART_NAN;
            int flags = 0;
            if (k >= 2) {
                const double x = g2w - Vk;                        // Eq. (11)
                N = x > 0.0 ? x : 0.0;
            } else {
                V = CUDART_NAN;
                flags |= DBW_FLAG_K1;
            }
            if (sh->t >= 1 && sh->has_last) {                     // Eq. (12)
                if (den > 0.0) L = L12;
                if (!(den > 0.0 && isfinite(L))) {
                    L = CUDART_NAN;
                    flags |= DBW_FLAG_L_SKIPPED;
                } else {
                    st->ringL[sh->cntL % DBW_DMAX] = L;
                    st->cntL = sh->cntL + 1;
                }
            }
            if (k >= 2) {
                st->ringV[sh->cntV % DBW_DMAX] = V;
                st->cntV = sh->cntV + 1;
                st->ringN[sh->cntN % DBW_DMAX] = N;
                st->cntN = sh->cntN + 1;
                st->N_last = N;
                st->V_last = V;
                st->has_last = 1;
            } else {
                st->N_last = CUDART_NAN;
                st->V_last = CUDART_NAN;
                st->has_last = 0;
            }
            st->c = sh->c + 1;
            const double vclock = sh->vclock + tsorted[k - 1];
            st->vclock = vclock;
            st->F_prev = sh->F_last;
            st->F_last = F;
            st->k_last = k;
            st->t = sh->t + 1;
            st->flags = sh->flags | flags;
            if (stats_out) {
                stats_out[DBW_STAT_K] = (double)k;
                stats_out[DBW_STAT_SS] = SS;
                stats_out[DBW_STAT_GBAR_SQ] = g2;
                stats_out[DBW_STAT_V] = V;
                stats_out[DBW_STAT_N] = N;
                stats_out[DBW_STAT_F] = F;
                stats_out[DBW_STAT_L] = L;
                stats_out[DBW_STAT_FLAGS] = (double)flags;
                stats_out[DBW_STAT_VCLOCK] = vclock;
            }
        }
    }
}

// T_ext (nullable): time estimates T^_k = T_ext[k-1] instead of S[k-1] / c; NaN in
// T_ext[0] means no estimate yet.
__global__ void __launch_bounds__(1024) choose_b_kernel(dbw_state* __restrict__ st, double lr, double beta,
                                                        int flags, int32_t* __restrict__ b_out,
                                                        double* __restrict__ ratio_out,
                                                        const double* __restrict__ T_ext) {
    grid_begin();
    __shared__ double mean_s[3];
    __shared__ int ready_s;
    __shared__ double best_r[32];
    __shared__ int best_k[32];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    __shared__ unsigned long long head_s[kHeadWords];
    const dbw_state* sh = stage_head(st, head_s);
    const int n = sh->n;
    if (n < 1 || n > DBW_NMAX || sh->D < 1 || sh->D > DBW_DMAX || sh->cntV < 0 || sh->cntN < 0 ||
        sh->cntL < 0 || sh->c < 0) {
        if (tid == 0) st->flags = sh->flags | DBW_FLAG_BAD_STATE;
        return;
    }
    const bool blind = (flags & DBW_CHOOSE_BLIND) != 0;
    // the three windows' rings, loaded by every thread at once (window_mean then sums
    // them in its fixed order from shared memory)
    __shared__ double ring_s[3][DBW_DMAX];
    for (int e = tid; e < 3 * DBW_DMAX; e += blockDim.x) {
        const int r = e / DBW_DMAX, i = e - r * DBW_DMAX;
        ring_s[r][i] = (r == 0 ? st->ringV : r == 1 ? st->ringN : st->ringL)[i];
    }
    __syncthreads();
    const double c = (double)sh->c;
    // this thread's first time estimate, while the windows are summed
    const double T_first = tid < n ? (T_ext ? T_ext[tid] : st->S[tid] / c) : 0.0;
    if (tid < 3) {
        // thread 0 the window of Eq. (13), 1 that of Eq. (14), 2 that of Eq. (15)
        const bool have_T = T_ext ? !isnan(T_ext[0]) : sh->c > 0;
        const bool windows = sh->cntV > 0 && sh->cntN > 0 && sh->cntL > 0 && sh->c > 0;
        if (!blind && windows)
            mean_s[tid] = window_mean(ring_s[tid], tid == 0 ? sh->cntV : tid == 1 ? sh->cntN : sh->cntL, sh->D);
        if (tid == 0) ready_s = blind ? have_T : windows && have_T;
    }
    __syncthreads();
    const int ready = ready_s;
    const double Vh = mean_s[0], Nh = mean_s[1];
    const double q = ((mean_s[2] * lr) * lr) / 2.0;
    // candidate of this thread: k = tid + 1
    double my_r = -CUDART_INF;
    int my_k = 0;   // 0 = not eligible
    for (int k = tid + 1; k <= n; k += blockDim.x) {
        double ratio = CUDART_NAN;
        bool elig = false;
        if (ready) {
            const double T = k == tid + 1 ? T_first : T_ext ? T_ext[k - 1] : st->S[k - 1] / c;   // T^_k
            if (blind) {
                ratio = (double)k / T;
                elig = true;
            } else {
                const double gain = ((lr - q) * Nh) - (q * (Vh / (double)k));   // Eq. (16)
                ratio = gain / T;
                elig = gain > 0.0;
            }
        }
        if (ratio_out) ratio_out[k - 1] = ratio;
        if (elig && (my_k == 0 || ratio > my_r || (ratio == my_r && k > my_k))) {
            my_r = ratio;
            my_k = k;
        }
    }
    // Eq. (18): lexicographic max of (eligible, ratio, k) across the CTA
    for (int o = 16; o > 0; o >>= 1) {
        const double r2 = __shfl_xor_sync(0xffffffffu, my_r, o);
        const int k2 = __shfl_xor_sync(0xffffffffu, my_k, o);
        if (k2 != 0 && (my_k == 0 || r2 > my_r || (r2 == my_r && k2 > my_k))) {
            my_r = r2;
            my_k = k2;
        }
    }
    if (lane == 0) {
        best_r[warp] = my_r;
        best_k[warp] = my_k;
    }
    __syncthreads();
    if (tid == 0) {
        int kstar = 0;
        double rbest = -CUDART_INF;
        for (int wv = 0; wv < (int)(blockDim.x >> 5); ++wv) {
            const int k2 = best_k[wv];
            const double r2 = best_r[wv];
            if (k2 != 0 && (kstar == 0 || r2 > rbest || (r2 == rbest && k2 > kstar))) {
                rbest = r2;
                kstar = k2;
            }
        }
        if (kstar == 0) kstar = n;                                // R3 / R7: k = n
        if (sh->t >= 2 && sh->F_last > beta * sh->F_prev && sh->k_last < n) {   // Eq. (19)
            const int kg = sh->k_last + 1;
            if (kg > kstar) kstar = kg;
        }
        if (kstar > n) kstar = n;
        st->k_next = kstar;
        *b_out = n - kstar;
    }
}

__global__ void state_init_kernel(dbw_state* st, int n, int D) {
    grid_begin();
    double* raw = reinterpret_cast<double*>(st);
    const int nwords = (int)(sizeof(dbw_state) / sizeof(double));
    for (int i = threadIdx.x; i < nwords; i += blockDim.x) raw[i] = 0.0;
    __syncthreads();
    if (threadIdx.x == 0) {
        st->n = n;
        st->D = D;
        st->k_next = n;
        st->F_last = CUDART_NAN;
        st->F_prev = CUDART_NAN;
        st->N_last = CUDART_NAN;
        st->V_last = CUDART_NAN;
    }
}

}  // namespace

cudaError_t launch_state_init(dbw_state* s, int n, int D, cudaStream_t st) {
    launch(state_init_kernel, 1, 256, 0, st, s, n, D);
    return cudaGetLastError();
}

cudaError_t launch_grad_stats(const double* partials, int n, const uint8_t* mask, const float* loss,
                              const double* tsorted, double lr, dbw_state* s, double* stats_out,
                              double* row_sqnorm, cudaStream_t st) {
    launch(grad_stats_kernel, n + 1, kRedThreads, 0, st, const_cast<double*>(partials), n, mask, loss, tsorted, lr, s,
                                                     stats_out, row_sqnorm);
    return cudaGetLastError();
}

cudaError_t launch_choose_b(dbw_state* s, double lr, double beta, int flags, int32_t* b_out,
                            double* ratio_out, const double* T_ext, cudaStream_t st) {
    // a thread per candidate k; the launch does not know the state's n
    launch(choose_b_kernel, 1, 1024, 0, st, s, lr, beta, flags, b_out, ratio_out, T_ext);
    return cudaGetLastError();
}

}  // namespace dbw
