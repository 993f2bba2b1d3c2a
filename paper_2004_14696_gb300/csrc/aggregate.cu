// Eqs. (3)-(4) fused with the gradient statistics of Sect. 3.1 in one pass over
// the received rows of G: masked column mean g_t, SGD step on w, and per-block
// pieces of sum_j ||g_j||^2, sum_{l,j} (G[j,l] - g_t[l])^2 and ||g_t||^2.
//
// HBM-bound: each received row is read once with 128-bit streaming loads and w
// is read and written once, so the algorithmic traffic is (k d + 2 d) * 4 bytes
// (+ d * 4 if g_t is stored).
//
// Two forms, with the same arithmetic per column and row:
//
// aggregate_kernel (d < kWideMinCols).  A warp owns a chunk of 256 columns for all rows, so
// the column reductions stay in its lanes' registers and nothing is shared between warps
// but the output.  Rows come through a ring of R = 4 slots of shared memory per warp that
// each lane fills and reads for itself with 16-byte asynchronous copies (two batches of two
// rows, each refilled once it is reduced): no barrier, and no registers held by loads in
// flight.  Loads to registers, two batches of two rows, ran at 18.1 / 76.7 / 26.1 / 43.7 us
// where this runs at 12.1 / 45.4 / 17.8 / 43.3 (k = 48, d = 203,530 / k = 192, d = 203,530 /
// k = 48, d = 500,000 / k = 12, d = 4,000,000).
//
// aggregate_wide_kernel (d >= kWideMinCols).  From HBM the order of the requests counts:
// warps that walk the rows on their own leave 1 KB pieces of thousands of rows open at a
// time.  Here a CTA owns 2048 columns; a producer thread streams them row by row, 8 KB per
// bulk copy, through a ring of 4 stages, and eight warps reduce 256 columns each.  us for
// (k = 48, d = 1e7) / (64 rows read, d = 1e7) / (k = 192, d = 3e7): 297 / 384 / 3277, the
// warp form 300 / 394 / 3404, the register form 331 / 428 / 3573; the last at 7.14 TB/s
// (of measured copy bandwidth: 1.05).  Below kWideMinCols a CTA has few chunks and the last
// round of them costs more.  Wide over narrow, everything received, at d = 2, 4, 6, 7, 7.9, 9 and 12
// million: k = 12 1.14, 1.06, 1.04, 1.04, 1.03, 1.06, 1.03; k = 48 1.06, 1.03, 1.01, 1.01, 1.005, 0.97,
// 0.99; k = 192 1.06, 1.01, 1.00, 0.98, 0.98, 0.98, 0.96.  Those calls find part of few rows in L2;
// with L2 flushed before each, d = 8.2e6 to 3e7, it is 0.87-1.01 at k = 1 .. 3, 0.91-1.07 at 4 .. 8 and
// 0.93-0.99 above.  (The dearest corner: one row of 8.2e6 that stays in L2, 28.6 us against 24.5.)
// Stages of two rows, 3 or 6 stages and 2 CTAs per SM were up to 4 % slower.
//
// Row norms.  The lanes' pieces of four rows are summed together: at each of the first two
// exchange steps a lane gives away half of the rows it holds, so four rows cost 6 shuffles
// instead of 20, and the four sums end in different lanes, which add them to the fp64
// accumulators in one instruction.  Each sum's tree is that of one butterfly per row.
//
// With DBW_ALL_ROW_NORMS the rows the mask leaves out are read too, after the
// received ones, for their squared norms only (Sect. 3.1's statistics still use
// the received rows alone); that adds (n - k) d * 4 bytes.  It is a separate
// instantiation of the kernel, so the default one is unchanged.
//
// Numerics.  Per column the warp keeps s1 = sum (x - c) and s2 = sum (x - c)^2 in
// fp32 with the shift c = the column's value in the first received row, so that
// sum_j (x_j - mean)^2 = s2 - s1^2 / k does not cancel.  Per-row squared norms
// are reduced across the warp in fp32 per chunk and accumulated in fp64 in shared
// memory (each row slot is owned by one warp, so no atomics); the column
// statistics are accumulated in fp64 per lane.  All reductions run in a fixed
// order, so results are deterministic for a given device.
#include "common.cuh"
#include "tc_ptx.cuh"

namespace dbw {

namespace {

constexpr int kThreads = 256;
constexpr int kWarps = kThreads / 32;
constexpr int VEC = 2;   // float4 per lane per row: chunk = 32 * VEC * 4 columns
constexpr int UB = 2;     // rows per batch
constexpr int NB = 2;     // batches in the ring
constexpr int R = UB * NB;     // rows per group: their norms are summed together
constexpr int kCtasPerSm = 3;
constexpr int kChunkCols = 32 * VEC * 4;
constexpr int kSlotFloats = kChunkCols;   // a ring slot: one row of a chunk
constexpr size_t kRingBytes = (size_t)kWarps * R * kSlotFloats * 4;
static_assert(R == 2 || R == 4 || R == 8 || R == 16, "the group sum halves R rows at a time");

__device__ __forceinline__ float4 ldg_stream(const float4* p) {
    float4 v;
    asm volatile("ld.global.nc.L1::no_allocate.L2::256B.v4.f32 {%0,%1,%2,%3}, [%4];"
                 : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
                 : "l"(p));
    return v;
}

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

__device__ __forceinline__ double warp_sum_d(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// Sums of R rows' lane pieces across the warp; lane l returns the sum of row l / (32 / R).
template <int N>
__device__ __forceinline__ float group_sum(float (&v)[N], int lane) {
    int half = 16;
#pragma unroll
    for (int rows = N; rows > 1; rows >>= 1, half >>= 1) {
        const bool up = (lane & half) != 0;   // keeps the upper half of the rows, gives the lower
#pragma unroll
        for (int i = 0; i < rows / 2; ++i) {
            const float keep = up ? v[i + rows / 2] : v[i];
            const float give = up ? v[i] : v[i + rows / 2];
            v[i] = keep + __shfl_xor_sync(0xffffffffu, give, half);
        }
    }
    float s = v[0];
#pragma unroll
    for (int o = 16 / N; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    return s;
}

// Column epilogue of a chunk: mean, SGD step, deviation sum, ||g_t||^2.
template <int V>
__device__ __forceinline__ void chunk_update(const float4 (&c)[V], const float4 (&s1)[V], const float4 (&s2)[V],
                                             int64_t col0, int64_t d, float inv_k, float lr, float* __restrict__ w,
                                             float* __restrict__ gbar, double& ss_acc, double& g2_acc) {
    float ss_chunk = 0.f, g2_chunk = 0.f;
#pragma unroll
    for (int v = 0; v < V; ++v) {
        const int64_t col = col0 + v * 128;
        if (col >= d) continue;
        float m[4], dev[4];
        const float* c4 = &c[v].x;
        const float* a4 = &s1[v].x;
        const float* b4 = &s2[v].x;
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            m[e] = c4[e] + a4[e] * inv_k;
            dev[e] = b4[e] - a4[e] * a4[e] * inv_k;
        }
        if (col + 3 < d) {
            float4 wv = *reinterpret_cast<const float4*>(w + col);
            wv.x = fmaf(-lr, m[0], wv.x); wv.y = fmaf(-lr, m[1], wv.y);
            wv.z = fmaf(-lr, m[2], wv.z); wv.w = fmaf(-lr, m[3], wv.w);
            *reinterpret_cast<float4*>(w + col) = wv;
            if (gbar) *reinterpret_cast<float4*>(gbar + col) = make_float4(m[0], m[1], m[2], m[3]);
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                ss_chunk += dev[e];
                g2_chunk = fmaf(m[e], m[e], g2_chunk);
            }
        } else {
            for (int e = 0; e < 4 && col + e < d; ++e) {
                w[col + e] = fmaf(-lr, m[e], w[col + e]);
                if (gbar) gbar[col + e] = m[e];
                ss_chunk += dev[e];
                g2_chunk = fmaf(m[e], m[e], g2_chunk);
            }
        }
    }
    ss_acc += (double)ss_chunk;
    g2_acc += (double)g2_chunk;
}

// Adds a row's columns to the shifted sums (``stats``: a received row) and to r its squares.
template <int V>
__device__ __forceinline__ void add_row(const float4 (&x)[V], const float4 (&c)[V], float4 (&s1)[V], float4 (&s2)[V],
                                        float& r, bool stats) {
#pragma unroll
    for (int v = 0; v < V; ++v) {
        if (stats) {   // rows read past the received ones add no statistics
            const float dx0 = x[v].x - c[v].x, dx1 = x[v].y - c[v].y;
            const float dx2 = x[v].z - c[v].z, dx3 = x[v].w - c[v].w;
            s1[v].x += dx0; s1[v].y += dx1; s1[v].z += dx2; s1[v].w += dx3;
            s2[v].x = fmaf(dx0, dx0, s2[v].x); s2[v].y = fmaf(dx1, dx1, s2[v].y);
            s2[v].z = fmaf(dx2, dx2, s2[v].z); s2[v].w = fmaf(dx3, dx3, s2[v].w);
        }
        r = fmaf(x[v].x, x[v].x, r); r = fmaf(x[v].y, x[v].y, r);
        r = fmaf(x[v].z, x[v].z, r); r = fmaf(x[v].w, x[v].w, r);
    }
}

// 16 bytes of this thread, global -> its own place in shared memory, without passing through
// registers; bytes past ``bytes`` (0..16) are zero and not read.
__device__ __forceinline__ void copy16(uint32_t dst, const float* src, uint32_t bytes) {
    asm volatile("cp.async.cg.shared.global.L2::256B [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(bytes) : "memory");
}
__device__ __forceinline__ void bulk_load(uint32_t dst, const float* src, uint32_t bytes, uint32_t bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
                 "l"(src), "r"(bytes), "r"(bar)
                 : "memory");
}
__device__ __forceinline__ void copy_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void copy_wait() {
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// One chunk of columns over all rows.  ``ring``: this lane's place in the warp's ring (slot
// r at ring + r * kSlotFloats, its float4 v at + v * 128).
template <bool kAllRows>
__device__ __forceinline__ void chunk_pass(const float* __restrict__ G, int64_t ld, int64_t d, int64_t col0, int lane,
                                           int k, int nrows, float inv_k, float lr, const int* __restrict__ sel,
                                           double* __restrict__ myrow, float* ring, float* __restrict__ w,
                                           float* __restrict__ gbar, double& ss_acc, double& g2_acc) {
    // this lane's columns: col0 + v * 128 .. +3, v < VEC; columns >= d read as zero
    uint32_t bytes[VEC];
#pragma unroll
    for (int v = 0; v < VEC; ++v) {
        const int64_t left = d - (col0 + v * 128);
        bytes[v] = left >= 4 ? 16u : left > 0 ? static_cast<uint32_t>(left) * 4u : 0u;
    }
    const float* Gc = G + col0;
    const uint32_t ring_s = static_cast<uint32_t>(__cvta_generic_to_shared(ring));
    auto fetch = [&](int p, int slot) {   // row p into a ring slot (nothing past the last row)
        if (p < nrows) {
            const float* rowp = Gc + (int64_t)sel[p] * ld;
#pragma unroll
            for (int v = 0; v < VEC; ++v)
                copy16(ring_s + (slot * kSlotFloats + v * 128) * 4, bytes[v] ? rowp + v * 128 : G, bytes[v]);
        }
    };
    float4 c[VEC], s1[VEC], s2[VEC];
    {   // row 0 of the received set gives the shift
        const float* rowp = Gc + (int64_t)sel[0] * ld;
#pragma unroll
        for (int v = 0; v < VEC; ++v) {
            c[v] = bytes[v] ? ldg_stream(reinterpret_cast<const float4*>(rowp + v * 128)) : make_float4(0.f, 0.f, 0.f, 0.f);
            if (bytes[v] < 16u) {
                if (bytes[v] < 8u) c[v].y = 0.f;
                if (bytes[v] < 12u) c[v].z = 0.f;
                c[v].w = 0.f;
            }
        }
    }
#pragma unroll
    for (int b = 0; b < NB; ++b) {
#pragma unroll
        for (int u = 0; u < UB; ++u) fetch(1 + b * UB + u, b * UB + u);
        copy_commit();
    }
    {
        float rn = 0.f;
#pragma unroll
        for (int v = 0; v < VEC; ++v) {
            s1[v] = make_float4(0.f, 0.f, 0.f, 0.f);
            s2[v] = make_float4(0.f, 0.f, 0.f, 0.f);
            rn += c[v].x * c[v].x + c[v].y * c[v].y + c[v].z * c[v].z + c[v].w * c[v].w;
        }
        rn = warp_sum(rn);
        if (lane == 0) myrow[0] += (double)rn;
    }
    for (int p0 = 1; p0 < nrows; p0 += R) {
        float rn[R];
#pragma unroll
        for (int b = 0; b < NB; ++b) {
            copy_wait<NB - 1>();   // this thread's copies of the oldest batch have landed
#pragma unroll
            for (int u = 0; u < UB; ++u) {
                const int p = p0 + b * UB + u;
                float r = 0.f;
                if (p < nrows) {
                    float4 x[VEC];
#pragma unroll
                    for (int v = 0; v < VEC; ++v)
                        x[v] = *reinterpret_cast<const float4*>(ring + (b * UB + u) * kSlotFloats + v * 128);
                    add_row<VEC>(x, c, s1, s2, r, !kAllRows || p < k);
                }
                rn[b * UB + u] = r;
            }
#pragma unroll
            for (int u = 0; u < UB; ++u) fetch(p0 + R + b * UB + u, b * UB + u);
            copy_commit();
        }
        const float mine = group_sum(rn, lane);
        const int p = p0 + lane / (32 / R);
        if (lane % (32 / R) == 0 && p < nrows) myrow[p] += (double)mine;
    }
    chunk_update<VEC>(c, s1, s2, col0, d, inv_k, lr, w, gbar, ss_acc, g2_acc);
}

// Reading order of the rows into sel [n]: the received ones, then (kAllRows) the others,
// each in increasing order; returns k.  kThreads threads of the block take part (tid <
// kThreads); ``bar`` is a barrier of exactly those threads.
template <bool kAllRows, class Bar>
__device__ __forceinline__ int reading_order(const uint8_t* __restrict__ mask, int n, int* sel, int* warp_cnt, Bar bar) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    // positions by ballots, 256 workers at a time; a worker the mask leaves out is parked at
    // the end of the list (its place from the back) until k is known
    int k = 0;
    for (int j0 = 0; j0 < n; j0 += kThreads) {
        const int j = j0 + tid;
        const bool on = j < n && mask[j] != 0;
        const unsigned bal = __ballot_sync(0xffffffffu, on);
        if (lane == 0) warp_cnt[warp] = __popc(bal);
        bar();
        int before = k;
        for (int q = 0; q < kWarps; ++q) {
            if (q < warp) before += warp_cnt[q];
            k += warp_cnt[q];
        }
        const int rank = before + __popc(bal & ((1u << lane) - 1u));   // received workers below j
        if (on) sel[rank] = j;
        else if (kAllRows && j < n) sel[n - 1 - (j - rank)] = j;
        bar();
    }
    if (kAllRows) {   // the parked ones are in decreasing order from position k
        const int others = n - k;
        for (int i = tid; i < others / 2; i += kThreads) {
            const int t = sel[k + i];
            sel[k + i] = sel[n - 1 - i];
            sel[n - 1 - i] = t;
        }
    }
    return k;
}

__device__ __forceinline__ void write_header(double* partials, int nblocks, int n, bool all_rows) {
    int64_t* hdr = reinterpret_cast<int64_t*>(partials);
    hdr[0] = kPartialsMagic;
    hdr[1] = nblocks;
    hdr[2] = n;
    hdr[3] = all_rows ? DBW_ALL_ROW_NORMS : 0;
}

// This block's pieces: the row norms (rowacc [kWarps][n], by reading position), then the
// two column sums.  Fixed-order reductions; the same threads and barrier as reading_order.
template <bool kAllRows, class Bar>
__device__ __forceinline__ void write_pieces(double* __restrict__ partials, int nblocks, int n, int nrows,
                                             const uint8_t* __restrict__ mask, const int* sel, const double* rowacc,
                                             double ss_acc, double g2_acc, double (*red)[kWarps], bool timed_out,
                                             Bar bar) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    ss_acc = warp_sum_d(ss_acc);
    g2_acc = warp_sum_d(g2_acc);
    if (lane == 0) {
        red[0][warp] = ss_acc;
        red[1][warp] = g2_acc;
    }
    double* vals = partials + kPartialsHeader + (n + 2);
    if (!kAllRows)
        for (int q = tid; q < n; q += kThreads)
            if (!mask[q]) vals[(int64_t)q * nblocks + blockIdx.x] = 0.0;
    bar();
    const double lost = __longlong_as_double(kPieceTimedOut);
    // rows are indexed by reading position in rowacc; scatter them to worker ids
    for (int p = tid; p < nrows; p += kThreads) {
        double t = 0.0;
        for (int wv = 0; wv < kWarps; ++wv) t += rowacc[(size_t)wv * n + p];
        vals[(int64_t)sel[p] * nblocks + blockIdx.x] = timed_out ? lost : t;
    }
    if (tid == 0) {
        double x = 0.0, y = 0.0;
        for (int wv = 0; wv < kWarps; ++wv) {
            x += red[0][wv];
            y += red[1][wv];
        }
        vals[(int64_t)n * nblocks + blockIdx.x] = timed_out ? lost : x;
        vals[(int64_t)(n + 1) * nblocks + blockIdx.x] = timed_out ? lost : y;
        if (blockIdx.x == 0) write_header(partials, nblocks, n, kAllRows);
    }
}

// kAllRows: also the squared norms of the rows the mask leaves out (DBW_ALL_ROW_NORMS).
template <bool kAllRows>
__global__ void __launch_bounds__(kThreads, kCtasPerSm) aggregate_kernel(
    const float* __restrict__ G, int64_t ld, int n, int64_t d, const uint8_t* __restrict__ mask,
    float lr, float* __restrict__ w, float* __restrict__ gbar, double* __restrict__ partials,
    int nblocks) {
    grid_begin();
    extern __shared__ __align__(16) double smem_d[];
    float* rings = reinterpret_cast<float*>(smem_d);   // [kWarps][R] ring slots
    double* rowacc = smem_d + kRingBytes / 8;          // [kWarps][n] fp64 row-norm pieces
    int* sel = reinterpret_cast<int*>(rowacc + (size_t)kWarps * n);
    __shared__ int warp_cnt[kWarps];
    __shared__ double red[2][kWarps];
    auto bar = [] { __syncthreads(); };

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int k = reading_order<kAllRows>(mask, n, sel, warp_cnt, bar);
    for (int i = tid; i < kWarps * n; i += kThreads) rowacc[i] = 0.0;
    __syncthreads();
    if (k == 0) {   // nothing received: leave w untouched, record empty pieces
        double* vals = partials + kPartialsHeader + (n + 2);
        for (int q = tid; q < n + 2; q += kThreads) vals[(int64_t)q * nblocks + blockIdx.x] = 0.0;
        if (blockIdx.x == 0 && tid == 0) write_header(partials, nblocks, n, kAllRows);
        return;
    }
    // rows read per chunk: the k received ones (their statistics), then with kAllRows
    // the n - k others (their squared norms only)
    const int nrows = kAllRows ? n : k;
    const float inv_k = 1.0f / (float)k;
    double* myrow = rowacc + (size_t)warp * n;
    float* ring = rings + (size_t)warp * R * kSlotFloats + lane * 4;

    double ss_acc = 0.0, g2_acc = 0.0;
    const int64_t nchunks = (d + kChunkCols - 1) / kChunkCols;
    const int64_t nwarps_total = (int64_t)nblocks * kWarps;
    for (int64_t chunk = (int64_t)blockIdx.x * kWarps + warp; chunk < nchunks; chunk += nwarps_total) {
        const int64_t col0 = chunk * kChunkCols + lane * 4;
        chunk_pass<kAllRows>(G, ld, d, col0, lane, k, nrows, inv_k, lr, sel, myrow, ring, w, gbar, ss_acc, g2_acc);
    }
    write_pieces<kAllRows>(partials, nblocks, n, nrows, mask, sel, rowacc, ss_acc, g2_acc, red, false, bar);
}

// ------------------------------------------------------------------ wide form
// Warps 0-7 reduce, warp 8's first lane produces.  A stage holds one row of the CTA's
// chunk; full[s] completes when its bytes have landed, empty[s] when the eight warps have
// read it.  Every wait is bounded (2 s).  A warp one of whose waits ran out leaves w and g_t as
// they are in that chunk and stops; it frees no further stage, so that the others either read
// rows that have landed or run out in turn.  The block's pieces then all say so (kPieceTimedOut).
// kTest: the instantiation of the tests of that path (see TestWaits).
constexpr int kWideVec = 2;                                // float4 per lane and row
constexpr int kWideCols = kWarps * 128 * kWideVec;
constexpr int kWideStages = 4;                                   // one row of a chunk each
constexpr int kWideGroup = 4;                                     // rows whose norms are summed together
constexpr int kWideThreads = kThreads + 32;
constexpr int kWideStageFloats = kWideCols;
constexpr size_t kWideRing = (size_t)kWideStages * kWideStageFloats * 4;

template <bool kAllRows, bool kTest = false>
__global__ void __launch_bounds__(kWideThreads, 3) aggregate_wide_kernel(
    const float* __restrict__ G, int64_t ld, int n, int64_t d, const uint8_t* __restrict__ mask,
    float lr, float* __restrict__ w, float* __restrict__ gbar, double* __restrict__ partials,
    int nblocks, TestWaits wt) {
    grid_begin();
    using namespace tcx;
    const uint64_t wait_ns = kTest ? wt.limit_ns : kWaitLimitNs;
    extern __shared__ __align__(128) double smem_w[];
    float* ring = reinterpret_cast<float*>(smem_w);
    double* rowacc = smem_w + kWideRing / 8;
    int* sel = reinterpret_cast<int*>(rowacc + (size_t)kWarps * n);
    __shared__ int warp_cnt[kWarps];
    __shared__ double red[2][kWarps];
    __shared__ __align__(8) uint64_t full_bar[kWideStages], empty_bar[kWideStages];
    __shared__ int k_s, abort_s;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    auto bar = [] { asm volatile("bar.sync 1, 256;" ::: "memory"); };   // the consumer warps
    if (tid == 0) {
        for (int s = 0; s < kWideStages; ++s) {
            mbar_init(smem_u32(full_bar + s), 1);
            mbar_init(smem_u32(empty_bar + s), kWarps);
        }
        abort_s = 0;
        fence_mbar_init();
    }
    if (warp < kWarps) {
        const int kk = reading_order<kAllRows>(mask, n, sel, warp_cnt, bar);
        for (int i = tid; i < kWarps * n; i += kThreads) rowacc[i] = 0.0;
        if (tid == 0) k_s = kk;
    }
    __syncthreads();
    const int k = k_s;
    if (k == 0) {
        double* vals = partials + kPartialsHeader + (n + 2);
        for (int q = tid; q < n + 2; q += kWideThreads) vals[(int64_t)q * nblocks + blockIdx.x] = 0.0;
        if (blockIdx.x == 0 && tid == 0) write_header(partials, nblocks, n, kAllRows);
        return;
    }
    const int nrows = kAllRows ? n : k;
    const int64_t nchunks = (d + kWideCols - 1) / kWideCols;
    volatile int* vabort = &abort_s;
    if (warp == kWarps) {
        if (lane == 0) {
            uint32_t it = 0;
            for (int64_t c = blockIdx.x; c < nchunks && !*vabort; c += nblocks) {
                const int64_t col0 = c * kWideCols, left = d - col0;
                const uint32_t bytes = left >= kWideCols ? kWideCols * 4u : (uint32_t)((left + 3) / 4) * 16u;
                for (int p = 0; p < nrows; ++p, ++it) {
                    const int s = it % kWideStages;
                    if (!mbar_wait(smem_u32(empty_bar + s), ((it / kWideStages) & 1) ^ 1, wait_ns)) {
                        *vabort = 1;
                        break;
                    }
                    if (kTest && blockIdx.x == 0 && it == wt.skip_stage) continue;
                    const uint32_t fb = smem_u32(full_bar + s);
                    mbar_expect_tx(fb, bytes);
                    bulk_load(smem_u32(ring + s * kWideCols), G + (int64_t)sel[p] * ld + col0, bytes, fb);
                }
            }
            // the last copies land before the shared memory is given up, whatever the warps do
            for (uint32_t q = it < kWideStages ? 0 : it - kWideStages; q < it; ++q)
                mbar_wait(smem_u32(full_bar + q % kWideStages), (q / kWideStages) & 1, wait_ns);
        }
        return;
    }
    const float inv_k = 1.0f / (float)k;
    double* myrow = rowacc + (size_t)warp * n;
    const float* mine = ring + warp * 128 * kWideVec + lane * 4;
    double ss_acc = 0.0, g2_acc = 0.0;
    uint32_t it = 0;
    bool dead = false;
    for (int64_t ch = blockIdx.x; ch < nchunks; ch += nblocks) {
        const int64_t col0 = ch * kWideCols + warp * 128 * kWideVec + lane * 4;
        const bool full = (ch + 1) * kWideCols <= d;
        float4 c[kWideVec], s1[kWideVec], s2[kWideVec];
#pragma unroll
        for (int v = 0; v < kWideVec; ++v) c[v] = s1[v] = s2[v] = make_float4(0.f, 0.f, 0.f, 0.f);
        for (int p0 = 0; p0 < nrows; p0 += kWideGroup) {
            float rn[kWideGroup];
#pragma unroll
            for (int h = 0; h < kWideGroup; ++h) {
                const int p = p0 + h;
                float r = 0.f;
                if (p < nrows) {
                    const int s = it % kWideStages;
                    if (!dead && !mbar_wait(smem_u32(full_bar + s), (it / kWideStages) & 1, wait_ns)) {
                        dead = true;
                        *vabort = 1;
                    }
                    ++it;
                    float4 x[kWideVec];
#pragma unroll
                    for (int v = 0; v < kWideVec; ++v)
                        x[v] = *reinterpret_cast<const float4*>(mine + s * kWideCols + v * 128);
                    __syncwarp();
                    if (lane == 0 && !dead) mbar_arrive(smem_u32(empty_bar + s));
                    if (!full) {   // columns >= d: row padding, or an earlier chunk's bytes
#pragma unroll
                        for (int v = 0; v < kWideVec; ++v) {
                            const int64_t col = col0 + v * 128;
                            if (col >= d) x[v].x = 0.f;
                            if (col + 1 >= d) x[v].y = 0.f;
                            if (col + 2 >= d) x[v].z = 0.f;
                            if (col + 3 >= d) x[v].w = 0.f;
                        }
                    }
                    if (p == 0) {
#pragma unroll
                        for (int v = 0; v < kWideVec; ++v) c[v] = x[v];
                    }
                    // row 0 is the shift itself: left out of the sums, where an infinity would leave a NaN
                    add_row<kWideVec>(x, c, s1, s2, r, p > 0 && (!kAllRows || p < k));
                }
                rn[h] = r;
            }
            const float tot = group_sum(rn, lane);
            const int p = p0 + lane / (32 / kWideGroup);
            if (lane % (32 / kWideGroup) == 0 && p < nrows) myrow[p] += (double)tot;
        }
        if (__any_sync(0xffffffffu, dead)) break;   // rows not read: no step from them
        chunk_update<kWideVec>(c, s1, s2, col0, d, inv_k, lr, w, gbar, ss_acc, g2_acc);
    }
    bar();
    write_pieces<kAllRows>(partials, nblocks, n, nrows, mask, sel, rowacc, ss_acc, g2_acc, red, *vabort != 0, bar);
}

size_t agg_smem_bytes(int n) { return kRingBytes + (size_t)kWarps * n * sizeof(double) + (size_t)n * sizeof(int); }
size_t wide_smem_bytes(int n) { return kWideRing + (size_t)kWarps * n * sizeof(double) + (size_t)n * sizeof(int); }

constexpr int64_t kWideMinCols = 8000000;
bool use_wide(int64_t d) { return d >= kWideMinCols; }

// The opt-in to shared memory belongs to the kernel and is shared by the host's threads: every
// call sets it to the need of the largest n, so that none lowers it between another's set and launch.
template <class Kern>
cudaError_t allow_smem(Kern kern, bool wide) {
    const size_t most = wide ? wide_smem_bytes(DBW_NMAX) : agg_smem_bytes(DBW_NMAX);
    return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)most);
}

// Co-resident CTAs of a kernel per SM with its dynamic shared memory.
template <class Kern>
int ctas_per_sm(Kern kern, bool wide, int n) {
    int per_sm = 0;
    allow_smem(kern, wide);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, wide ? kWideThreads : kThreads,
                                                  wide ? wide_smem_bytes(n) : agg_smem_bytes(n));
    return per_sm < 1 ? 1 : per_sm;
}

}  // namespace

AggGeometry agg_geometry(int n, int64_t d) {
    AggGeometry g;
    // both instantiations of a kernel have the same launch shape; the default one sets the grid
    const bool wide = use_wide(d);
    const int per_sm = wide ? ctas_per_sm(aggregate_wide_kernel<false>, true, n) : ctas_per_sm(aggregate_kernel<false>, false, n);
    const int64_t cols = wide ? kWideCols : kChunkCols * kWarps;   // columns of a CTA's chunks
    const int64_t need = (d + cols - 1) / cols;
    int64_t blocks = (int64_t)sm_count() * per_sm;
    if (blocks > need) blocks = need;
    if (blocks < 1) blocks = 1;
    g.blocks = (int)blocks;
    g.rows_stride = n + 2;
    g.bytes = (size_t)kPartialsHeader * sizeof(int64_t) + (size_t)(n + 2) * (blocks + 1) * sizeof(double);
    return g;
}

namespace {
template <bool kAllRows>
cudaError_t launch_aggregate_t(const float* G, int64_t ld, int n, int64_t d, const uint8_t* mask, float lr,
                               float* w, float* gbar, double* partials, const AggGeometry& g, cudaStream_t st) {
    const bool wide = use_wide(d);
    // A grid of several CTAs per SM must not be set up early: CTAs placed while other kernels
    // still hold an SM find its shared memory configured for those, fewer fit, and the rest of
    // this grid becomes a second round (n = 64, d = 1e7 in a row: 395 us, early 523).
    const bool early = g.blocks <= sm_count();
    if (!wide) {
        const cudaError_t e = allow_smem(aggregate_kernel<kAllRows>, false);
        if (e != cudaSuccess) return e;
        launch_when(early, aggregate_kernel<kAllRows>, g.blocks, kThreads, agg_smem_bytes(n), st, G, ld, n, d, mask, lr, w,
                    gbar, partials, g.blocks);
        return cudaGetLastError();
    }
    const TestWaits wt = take_test_waits();
    auto kern = wt.skip_stage >= 0 ? aggregate_wide_kernel<kAllRows, true> : aggregate_wide_kernel<kAllRows>;
    const cudaError_t e = allow_smem(kern, true);
    if (e != cudaSuccess) return e;
    launch_when(early, kern, g.blocks, kWideThreads, wide_smem_bytes(n), st, G, ld, n, d, mask, lr, w, gbar, partials,
                g.blocks, wt);
    return cudaGetLastError();
}
}  // namespace

cudaError_t launch_aggregate(const float* G, int64_t ld, int n, int64_t d, const uint8_t* mask,
                             float lr, float* w, float* gbar, int flags, double* partials, const AggGeometry& g,
                             cudaStream_t st) {
    if (flags & DBW_ALL_ROW_NORMS)
        return launch_aggregate_t<true>(G, ld, n, d, mask, lr, w, gbar, partials, g, st);
    return launch_aggregate_t<false>(G, ld, n, d, mask, lr, w, gbar, partials, g, st);
}

}  // namespace dbw
