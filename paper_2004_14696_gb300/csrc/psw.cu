// Push-and-wait clock and the time estimator of Eq. (17) (Sect. 2, 3.2).
//
// The state is one device buffer: a dbw_psw_header, the workers' residual busy
// times and pending samples, the cell table of Eq. (17) (per (h, i): a sum of
// samples in int64 fixed point, so that concurrent adds are exact and their
// order does not matter, and a count), the fitted cells, the dual variables of
// the previous fit (warm start) and the solver's scratch.
//
// The fit (fp32: on this part a dependent fp64 operation costs ~14x its fp32
// latency, and the pool-adjacent-violators chains are sequential) runs in one CTA
// over the rows whose diagonal cell has samples (group rows; a row's observed ranks
// are a prefix, so the order of Eq. (17) among their observed cells is generated by
// chains over observed cells only).  Each group row is a chain of the first family,
// each column over the group rows one of the second, their diagonal cells the third.
// A group table that fits in shared memory is fitted there, a chain per group of lanes
// (psw_fit_shared_kernel); a larger one in the state buffer, a chain split over up to
// eight threads whose block stacks are then merged (psw_estimate_kernel).
// Each projection is weighted pool-adjacent-violators with the sample counts as
// weights; Dykstra's increments p_f are kept as dual variables lambda_f = w p_f
// between calls (warm start).
//
// Exact block means.  The solution of Eq. (17) is constant on blocks, and each
// block's value is the count-weighted mean of its samples.  Once the fp32 sweeps
// have converged, one more sweep records which cells every projection pooled (chain
// neighbours left with the same value), and the union of those poolings gives the
// blocks.  Each block's mean is then formed from the exact int64 cell sums in fp64;
// neighbouring blocks that still break the order are merged (a bounded number of
// rounds, else the fp32 values stand and DBW_PSW_UNPOLISHED is raised).
//
// Every other diagonal cell is the pooled column mean, made nondecreasing (PAVA in
// fp64) and clipped to the bounds the fitted cells place on it.  Compiled with
// -fmad=false so that the pooling arithmetic rounds as written.
#include <limits.h>
#include <math.h>
#include <math_constants.h>

#include "common.cuh"

namespace dbw {

namespace {

constexpr double kUnit = 1.0 / 4294967296.0;   // 2^-32 per unit of the cell sums
constexpr double kMaxSample = 2147483648.0;     // 2^31: samples are clamped to [0, 2^31)
constexpr int kThreads = 1024;
constexpr size_t kHeaderBytes = 256;
constexpr float kMinTol = 1e-6f;                 // the fit runs in fp32: tolerances below its resolution are raised

struct Layout {
    size_t r, pend, pendv, sum, cnt, x, lam, w, bm, bw, bl, bp, ab, nbk, mv, rows, isrow, mu, par, root, csum, ccnt,
        xd, fd, bytes;
};

inline size_t up256(size_t b) { return (b + 255) / 256 * 256; }

// Threads of the fit: four per column while that stays within 512 threads, else two
// (and up to kMaxParts per row or diagonal chain), at most 1024.  Measured: four per
// column is faster up to n = 128; beyond 512 threads the registers per thread halve.
inline int fit_threads(int n) {
    int t = (4 * n + 31) / 32 * 32;
    if (t > 512) t = (2 * n + 31) / 32 * 32;
    return t < kThreads ? t : kThreads;
}

Layout layout(int n) {
    const size_t nn = static_cast<size_t>(n) * n;
    Layout L;
    size_t cur = kHeaderBytes;
    auto take = [&](size_t bytes) {
        const size_t at = cur;
        cur += up256(bytes);
        return at;
    };
    L.r = take(n * 8);
    L.pend = take(n * 8);
    L.pendv = take(n * 8);
    L.sum = take(nn * 8);
    L.cnt = take(nn * 4);
    L.x = take(nn * 4);
    L.lam = take(3 * nn * 4);
    L.w = take(nn * 4);
    const size_t nt = static_cast<size_t>(n) * fit_threads(n);   // n entries for each of T threads
    L.bm = take(nt * 4);
    L.bw = take(nt * 4);
    L.bl = take(nt * 4);
    L.bp = take(nt * 4);                                   // block start positions (split chains)
    L.ab = take(nt * 4);                                   // part whose merged block absorbed the block, or -1
    L.nbk = take(static_cast<size_t>(fit_threads(n)) * 4);        // block count of each thread's stack
    L.mv = take(static_cast<size_t>(fit_threads(n)) * 4);         // final values of the merged blocks
    L.rows = take(n * 4);
    L.isrow = take(n * 4);
    L.mu = take(n * 8);
    L.par = take(nn * 4);                                  // union-find parent of each group cell
    L.root = take(nn * 4);                                 // its block (root cell) in the current round
    L.csum = take(nn * 8);                                 // per block: exact sum of its cells' sums
    L.ccnt = take(nn * 4);                                 //            and of their counts
    L.xd = take(nn * 8);                                   // fp64 value of each fitted cell (its block's mean)
    L.fd = take(2 * static_cast<size_t>(n) * 8);           // fp64 PAVA stack of the free diagonal cells
    L.bytes = cur;
    return L;
}

struct View {
    dbw_psw_header* hdr;
    double *r, *pendv, *mu, *xd, *fd;
    float *x, *lam, *w, *bm, *bw, *mv;
    int32_t *pend, *cnt, *bl, *bp, *ab, *nbk, *rows, *isrow, *par, *root, *ccnt;
    unsigned long long *sum, *csum;
};

__host__ __device__ inline View view(char* base, const Layout& L) {
    View v;
    v.hdr = reinterpret_cast<dbw_psw_header*>(base);
    v.r = reinterpret_cast<double*>(base + L.r);
    v.pend = reinterpret_cast<int32_t*>(base + L.pend);
    v.pendv = reinterpret_cast<double*>(base + L.pendv);
    v.sum = reinterpret_cast<unsigned long long*>(base + L.sum);
    v.cnt = reinterpret_cast<int32_t*>(base + L.cnt);
    v.x = reinterpret_cast<float*>(base + L.x);
    v.lam = reinterpret_cast<float*>(base + L.lam);
    v.w = reinterpret_cast<float*>(base + L.w);
    v.bm = reinterpret_cast<float*>(base + L.bm);
    v.bw = reinterpret_cast<float*>(base + L.bw);
    v.bl = reinterpret_cast<int32_t*>(base + L.bl);
    v.bp = reinterpret_cast<int32_t*>(base + L.bp);
    v.ab = reinterpret_cast<int32_t*>(base + L.ab);
    v.nbk = reinterpret_cast<int32_t*>(base + L.nbk);
    v.mv = reinterpret_cast<float*>(base + L.mv);
    v.rows = reinterpret_cast<int32_t*>(base + L.rows);
    v.isrow = reinterpret_cast<int32_t*>(base + L.isrow);
    v.mu = reinterpret_cast<double*>(base + L.mu);
    v.par = reinterpret_cast<int32_t*>(base + L.par);
    v.root = reinterpret_cast<int32_t*>(base + L.root);
    v.csum = reinterpret_cast<unsigned long long*>(base + L.csum);
    v.ccnt = reinterpret_cast<int32_t*>(base + L.ccnt);
    v.xd = reinterpret_cast<double*>(base + L.xd);
    v.fd = reinterpret_cast<double*>(base + L.fd);
    return v;
}

__global__ void psw_init_kernel(char* base, Layout L, int n) {
    grid_begin();
    View v = view(base, L);
    if (threadIdx.x == 0) {
        dbw_psw_header* h = v.hdr;
        h->n = n;
        h->h = n;
        h->sweeps = 0;
        h->flags = 0;
        h->vclock = 0.0;
        h->unit = kUnit;
        h->iterations = 0;
        h->off_r = static_cast<int64_t>(L.r);
        h->off_pend = static_cast<int64_t>(L.pend);
        h->off_pendv = static_cast<int64_t>(L.pendv);
        h->off_sum = static_cast<int64_t>(L.sum);
        h->off_cnt = static_cast<int64_t>(L.cnt);
        h->off_x = static_cast<int64_t>(L.x);
        for (int q = 0; q < 6; ++q) h->reserved[q] = 0;
    }
}

__global__ void psw_arrivals_kernel(const char* base, Layout L, int n, const double* __restrict__ omega,
                                    double* __restrict__ e) {
    grid_begin();
    const double* r = reinterpret_cast<const double*>(base + L.r);
    for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < n; j += gridDim.x * blockDim.x) e[j] = r[j] + omega[j];
}

__device__ inline void add_sample(View& v, int n, int h, int i, double val) {
    double c = val;
    if (!(c >= 0.0 && c < kMaxSample)) {
        atomicOr(&v.hdr->flags, DBW_PSW_RANGE);
        c = c >= kMaxSample ? kMaxSample - kUnit : 0.0;
    }
    const long long q = llrint(c / kUnit);
    const size_t cell = static_cast<size_t>(h - 1) * n + (i - 1);
    atomicAdd(v.sum + cell, static_cast<unsigned long long>(q));
    atomicAdd(v.cnt + cell, 1);
}

// One thread per position p of the arrival order (n <= 1024): worker j = order[p].
__global__ void __launch_bounds__(kThreads) psw_record_kernel(char* base, Layout L, int n,
                                                              const int32_t* __restrict__ order,
                                                              const double* __restrict__ tsorted,
                                                              const int32_t* __restrict__ kp) {
    grid_begin();
    __shared__ int warp_tot[32];
    View v = view(base, L);
    int k = *kp;
    k = k < 1 ? 1 : (k > n ? n : k);
    const double T = tsorted[k - 1];
    const int h = v.hdr->h;
    const int p = threadIdx.x, lane = p & 31, warp = p >> 5;
    int j = -1;
    double rj = 0.0;
    bool comp = false;
    if (p < n) {
        j = order[p];
        rj = v.r[j];
        comp = rj < T;   // free before w_{t+1} is pushed: computes on w_t
    }
    const unsigned bal = __ballot_sync(0xffffffffu, comp);
    if (lane == 0) warp_tot[warp] = __popc(bal);
    __syncthreads();
    if (p < n) {
        int rank = __popc(bal & ((1u << lane) - 1u)) + 1;
        for (int q = 0; q < warp; ++q) rank += warp_tot[q];
        // a sample of an older iteration reaches the PS when worker j becomes free
        if (v.pend[2 * j] != 0 && rj <= T) {
            add_sample(v, n, v.pend[2 * j], v.pend[2 * j + 1], v.pendv[j]);
            v.pend[2 * j] = 0;
        }
        if (comp) {
            const double e = tsorted[p];
            if (e <= T) {
                add_sample(v, n, h, rank, e);
            } else {
                v.pend[2 * j] = h;
                v.pend[2 * j + 1] = rank;
                v.pendv[j] = e;
            }
            const double left = e - T;
            v.r[j] = left > 0.0 ? left : 0.0;
        } else {
            v.r[j] = rj - T;
        }
    }
    __syncthreads();
    if (p == 0) {
        v.hdr->h = k;
        v.hdr->vclock = v.hdr->vclock + T;
        v.hdr->iterations += 1;
    }
}

// One Dykstra projection: nch chains of length len,
// position q of chain ch is cell cellf(ch, q) (a position whose weight is 0 has no
// samples and is skipped).  Every thread of the block must call it (it has two
// barriers).  Each chain gets P = min(T / nch, kMaxParts, len) threads.
//  1) Thread (ch, part) pools the positions [part len / P, (part + 1) len / P) into
//     its own block stack: weighted sum, weight, length, first position, absorber
//     (-1); entry e of thread t at e * T + t.
//  2) The chain's first thread merges the parts from left to right without moving
//     their blocks.  Part p's blocks are pushed, in order, on top of everything to
//     their left, with the pooling rule of pool-adjacent-violators: a block pools with
//     the top while the top's mean is larger.  What part p's first blocks pool into
//     becomes its merged block M_p, placed before part p's surviving blocks, and the
//     blocks and merged blocks it took in record p as their absorber.  Once a pushed
//     block of part p pools with nothing, the rest of part p survive: a part's blocks
//     increase.  This gives the blocks of pooling the positions one by one, since the
//     weighted isotonic regression is unique.  The final value of every merged block
//     (its own, or its absorber's) goes to mv.
//  3) Every thread assigns its positions. A surviving block gives its mean, or z for a
//     block that was never pooled. An absorbed block gives its absorber's final value.
// Returns the thread's largest |change of x|.
constexpr int kMaxParts = 8;

template <class CellF>
__device__ float split_chain_phase(float* __restrict__ X, float* __restrict__ PF, const float* __restrict__ W,
                                   CellF cellf, int nch, int len, float* __restrict__ bs, float* __restrict__ bw,
                                   int* __restrict__ bl, int* __restrict__ bp, int* __restrict__ ab,
                                   int* __restrict__ nbk, float* __restrict__ mv, int T) {
    const int tid = threadIdx.x;
    int P = nch > 0 ? T / nch : 1;
    P = P < 1 ? 1 : (P > kMaxParts ? kMaxParts : P);
    P = P > len ? (len > 0 ? len : 1) : P;
    const bool active = nch > 0 && len > 0 && tid < nch * P;
    const int ch = tid / P, part = tid % P;
    const int t0 = tid - part;
    const int q0 = static_cast<int>(static_cast<long long>(part) * len / P);
    const int q1 = static_cast<int>(static_cast<long long>(part + 1) * len / P);
    // 1) pool this part's positions.  The top block stays in registers (ts, tw, tl, tp);
    //    entries below it are in the stack, which a push appends to and a pool pops from.
    if (active) {
        int nb = 0;   // blocks, the top included
        float ts = 0.f, tw = 0.f;
        int tl = 0, tp = 0;
        // the next position's cell values are loaded while this one pools
        float nw = 0.f, nz = 0.f;
        if (q0 < q1) {
            const int c = cellf(ch, q0);
            nw = W[c];
            nz = X[c] + PF[c];
        }
        for (int q = q0; q < q1; ++q) {
            float ww = nw;
            const float z = nz;
            if (q + 1 < q1) {
                const int cn = cellf(ch, q + 1);
                nw = W[cn];
                nz = X[cn] + PF[cn];
            }
            if (!(ww > 0.f)) continue;
            float sm = z * ww;
            int l = 1, st = q;
            while (nb > 0 && ts * ww > sm * tw) {   // earlier mean > this mean
                sm = ts + sm;
                ww = tw + ww;
                l += tl;
                st = tp;
                --nb;
                if (nb > 0) {
                    const int e = (nb - 1) * T + tid;
                    ts = bs[e];
                    tw = bw[e];
                    tl = bl[e];
                    tp = bp[e];
                }
            }
            if (nb > 0) {   // the old top goes to the stack
                const int e = (nb - 1) * T + tid;
                bs[e] = ts;
                bw[e] = tw;
                bl[e] = tl;
                bp[e] = tp;
                ab[e] = -1;
            }
            ts = sm;
            tw = ww;
            tl = l;
            tp = st;
            ++nb;
        }
        if (nb > 0) {
            const int e = (nb - 1) * T + tid;
            bs[e] = ts;
            bw[e] = tw;
            bl[e] = tl;
            bp[e] = tp;
            ab[e] = -1;
        }
        nbk[tid] = nb;
    }
    __syncthreads();
    // 2) the chain's first thread merges the parts
    if (active && part == 0 && P > 1) {
        int lo[kMaxParts], hi[kMaxParts], mabs[kMaxParts];
        float msm[kMaxParts], mww[kMaxParts];
        bool mhas[kMaxParts];
        for (int q = 0; q < P; ++q) {
            lo[q] = 0;
            hi[q] = nbk[t0 + q];
            mhas[q] = false;
            mabs[q] = -1;
            msm[q] = 0.f;
            mww[q] = 0.f;
        }
        for (int p = 1; p < P; ++p) {
            const int tp = t0 + p;
            bool acc = false;
            float csm = 0.f, cww = 0.f;
            int e = 0;
            while (e < hi[p]) {
                const float bsm = bs[e * T + tp], bww = bw[e * T + tp];
                if (acc) {
                    if (!(csm * bww > bsm * cww)) break;   // M_p's mean <= this block's: the rest survive
                    csm += bsm;
                    cww += bww;
                } else {
                    csm = bsm;
                    cww = bww;
                }
                // pool with the top of everything to the left while its mean is larger
                bool pooled = false;
                for (;;) {
                    int zq = p - 1;
                    while (zq >= 0 && hi[zq] <= lo[zq] && !(mhas[zq] && mabs[zq] < 0)) --zq;
                    if (zq < 0) break;
                    if (hi[zq] > lo[zq]) {   // top: zone zq's last surviving block
                        const int te = (hi[zq] - 1) * T + t0 + zq;
                        if (!(bs[te] * cww > csm * bw[te])) break;
                        csm += bs[te];
                        cww += bw[te];
                        ab[te] = p;
                        --hi[zq];
                    } else {                 // top: zone zq's merged block
                        if (!(msm[zq] * cww > csm * mww[zq])) break;
                        csm += msm[zq];
                        cww += mww[zq];
                        mabs[zq] = p;
                    }
                    pooled = true;
                }
                if (!acc && !pooled) break;   // part p's first block pooled with nothing: all of part p survives
                ab[e * T + tp] = p;
                acc = true;
                ++e;
            }
            lo[p] = e;
            if (acc) {
                mhas[p] = true;
                msm[p] = csm;
                mww[p] = cww;
            }
        }
        // final value of each merged block: its own, or that of the block that took it in
        float fin[kMaxParts];
        for (int q = P - 1; q >= 1; --q) {
            if (!mhas[q]) continue;
            fin[q] = mabs[q] < 0 ? msm[q] / mww[q] : fin[mabs[q]];
            mv[t0 + q] = fin[q];
        }
    }
    __syncthreads();
    // 3) assign this part's positions
    float moved = 0.f;
    if (active) {
        const int nb = nbk[tid];
        int b = 0;
        int next = nb > 1 ? bp[T + tid] : INT_MAX;
        for (int q = q0; q < q1 && b < nb; ++q) {
            const int c = cellf(ch, q);
            if (!(W[c] > 0.f)) continue;
            while (q >= next) {
                ++b;
                next = b + 1 < nb ? bp[(b + 1) * T + tid] : INT_MAX;
            }
            const int e = b * T + tid;
            const float old = X[c];
            const float z = old + PF[c];
            const int who = ab[e];
            const float v = who >= 0 ? mv[t0 + who] : (bl[e] == 1 ? z : bs[e] / bw[e]);
            PF[c] = z - v;
            X[c] = v;
            moved = fmaxf(moved, fabsf(v - old));
        }
    }
    return moved;
}

__device__ float block_max(float v, float* red) {
    for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    __syncthreads();
    if (lane == 0) red[warp] = v;
    __syncthreads();
    float m = red[0];
    for (int q = 1; q < static_cast<int>(blockDim.x >> 5); ++q) m = fmaxf(m, red[q]);
    return m;
}

// ------------------------------------------------------------ blocks of the solution
// Union-find over cell indices, lock-free: a root is hooked under a smaller root with
// atomicCAS, so parent[x] <= x always holds and every find ends.
__device__ __forceinline__ int uf_find(volatile int32_t* par, int x) {
    for (;;) {
        const int p = par[x];
        if (p == x) return x;
        const int gp = par[p];
        if (gp != p) par[x] = gp;   // path halving: gp is still an ancestor of x
        x = p;
    }
}

__device__ __forceinline__ void uf_union(int32_t* par, int a, int b) {
    for (int guard = 0; guard < (1 << 22); ++guard) {   // each failed hook means another union succeeded
        a = uf_find(par, a);
        b = uf_find(par, b);
        if (a == b) return;
        if (a < b) {
            const int t = a;
            a = b;
            b = t;
        }
        if (atomicCAS(&par[a], a, b) == a) return;
    }
}

// f(prev, c) for every pair of consecutive observed cells of the nch chains (prev
// before c in chain order), with the threads split over the chains as in
// split_chain_phase; the pair across a part boundary goes to the later part.
template <class CellF, class EdgeF>
__device__ void for_chain_edges(const float* __restrict__ W, CellF cellf, int nch, int len, int T, EdgeF f) {
    const int tid = threadIdx.x;
    int P = nch > 0 ? T / nch : 1;
    P = P < 1 ? 1 : (P > kMaxParts ? kMaxParts : P);
    P = P > len ? (len > 0 ? len : 1) : P;
    if (!(nch > 0 && len > 0 && tid < nch * P)) return;
    const int ch = tid / P, part = tid % P;
    const int q0 = static_cast<int>(static_cast<long long>(part) * len / P);
    const int q1 = static_cast<int>(static_cast<long long>(part + 1) * len / P);
    int prev = -1;
    for (int q = q0 - 1; q >= 0; --q) {
        const int c = cellf(ch, q);
        if (W[c] > 0.f) {
            prev = c;
            break;
        }
    }
    for (int q = q0; q < q1; ++q) {
        const int c = cellf(ch, q);
        if (!(W[c] > 0.f)) continue;
        if (prev >= 0) f(prev, c);
        prev = c;
    }
}

// Dykstra sweeps over the group cells.  X, P0..P2, W address the cells through
// idx(a, i) (group row a, column i); bs .. mv are the chain-splitting scratch of
// split_chain_phase.
template <class Idx>
__device__ int dykstra_sweeps(float* X, float* P0, float* P1, float* P2, const float* W, Idx idx, const int32_t* rows,
                              int m, int n, float* bs, float* bw, int* bl, int* bp, int* ab, int* nbk, float* mv, int T,
                              float tol_abs, int max_sweeps, float* red, bool* converged) {
    int sweeps = 0;
    *converged = false;
    while (sweeps < max_sweeps) {
        ++sweeps;
        float moved = 0.f;
        // each group row increasing in k
        moved = fmaxf(moved, split_chain_phase(X, P0, W, [=](int a, int q) { return idx(a, q); }, m, n, bs, bw, bl, bp,
                                               ab, nbk, mv, T));
        __syncthreads();
        // each column decreasing in h over the group rows
        moved = fmaxf(moved, split_chain_phase(X, P1, W, [=](int i, int q) { return idx(m - 1 - q, i); }, n, m, bs, bw,
                                               bl, bp, ab, nbk, mv, T));
        __syncthreads();
        // the group rows' diagonal cells increasing in h
        moved = fmaxf(moved, split_chain_phase(X, P2, W, [=](int, int q) { return idx(q, rows[q] - 1); }, 1, m, bs, bw,
                                               bl, bp, ab, nbk, mv, T));
        // a sweep moves a cell by at most the sum of its three phase moves
        if (block_max(moved, red) * 3.f <= tol_abs) {
            *converged = true;
            break;
        }
    }
    return sweeps;
}

// One more Dykstra sweep after convergence, recording the blocks: after each
// projection, chain neighbours left with the same value (one pooled block, or tied
// blocks) are joined in par.
template <class Idx>
__device__ void record_sweep(float* X, float* P0, float* P1, float* P2, const float* W, Idx idx, const int32_t* rows,
                             int m, int n, float* bs, float* bw, int* bl, int* bp, int* ab, int* nbk, float* mv, int T,
                             int32_t* par) {
    auto rowf = [=](int a, int q) { return idx(a, q); };
    auto colf = [=](int i, int q) { return idx(m - 1 - q, i); };
    auto diagf = [=](int, int q) { return idx(q, rows[q] - 1); };
    auto join = [=](int a, int b) {
        if (X[a] == X[b]) uf_union(par, a, b);
    };
    split_chain_phase(X, P0, W, rowf, m, n, bs, bw, bl, bp, ab, nbk, mv, T);
    __syncthreads();
    for_chain_edges(W, rowf, m, n, T, join);
    __syncthreads();
    split_chain_phase(X, P1, W, colf, n, m, bs, bw, bl, bp, ab, nbk, mv, T);
    __syncthreads();
    for_chain_edges(W, colf, n, m, T, join);
    __syncthreads();
    split_chain_phase(X, P2, W, diagf, 1, m, bs, bw, bl, bp, ab, nbk, mv, T);
    __syncthreads();
    for_chain_edges(W, diagf, 1, m, T, join);
    __syncthreads();
}

constexpr int kFixRounds = 32;   // merging rounds of the exact block means

// ------------------------------------------------------------ the fit in shared memory
// The fit of a group table that fits in shared memory (72 rows at n = 96, 26 at 256, 17 at 384, 12
// at 512, 5 at 1024; the form above serves larger ones, at its own time: with 40 to 51 rows at
// n = 256 1.7-7.5 ms).  A sweep is a chain of dependent accesses, so latency is its
// time: there, with the table and the block stacks in the state buffer and chains split over
// at most eight threads whose stacks one thread merges, a sweep of 23 rows x 256 columns took
// 75-85 us and a whole fit of 19 / 43 / 61 sweeps 1.9 / 3.8 / 5.1 ms; here 15-18 us and
// 0.45 / 0.96 / 1.20 ms.  (A cluster of 2 or 4 CTAs, each projecting its share of the rows and
// columns into every CTA's copy of the table, took 0.94-1.02 and 0.90-1.02 of that: a phase is its
// longest chain, not the number of them.)
//
// The observed cells of every chain are listed once.  A chain belongs to a group of g lanes of
// a warp (g as large as the family's chains leave, at most 32).  Each lane pools its run of the
// chain by pool-adjacent-violators; then neighbouring runs, pairs of runs, ... are joined at
// their boundary in log2(g) steps: while the block before a boundary has a larger mean than the
// one after it, they pool, and the pooled block pools on with its neighbours on both sides.  The
// weighted isotonic regression is unique, so the blocks are those of the sequential scan.
// A block [s, e] of chain positions keeps its sum and weight at s, LK[s] = e and LK[e] = s; any
// other position p of it has LK[p] < p, so p starts a block iff LK[p] >= p.
struct SharedFit {
    int n, m, RS, MS, T;        // RS, MS: strides of a row's and a column's list
    float *X, *P0, *P1, *W;     // fitted cells, duals of the row and column chains, weights; cell (a, i) at a RS + i + i / 32
    float* P2;                  // [m] dual of the diagonal chain
    float *SM, *SW;             // block sums and weights of the current family's chains
    unsigned short* LK;
    unsigned short *rl, *cl, *dl;   // listed cells of each row (by increasing k), column (decreasing h), diagonal
    unsigned short *rc, *cc;    // their numbers
    unsigned short* par;        // union-find parents
    int *rows, *isrow;
    double* mu;
    int dc;
};
__host__ __device__ inline int fit_row_stride(int n) { return n + (n >> 5); }
__host__ __device__ inline size_t fit_slots(int n, int m) {   // of SM, SW, LK: both families' lists
    const size_t a = static_cast<size_t>(m) * fit_row_stride(n), b = static_cast<size_t>(n) * (m | 1);
    return ((a > b ? a : b) + 3) / 4 * 4;
}
__host__ __device__ inline size_t fit_shared_fixed(int n) {
    return (static_cast<size_t>(n) * (8 + 4 + 4 + 4 + 2 + 2 + 2) + 64) / 16 * 16;
}
// X, P0, P1, W, SM, SW; LK, par, the row and column lists
__host__ __device__ inline size_t fit_shared_bytes(int n, int m) {
    return fit_shared_fixed(n) + fit_slots(n, m) * (6 * 4 + 4 * 2);
}
inline int fit_shared_threads(int n) { return n < 32 ? 32 * ((n + 1) / 2 * 2) : 1024; }

__device__ __forceinline__ int fit_cell(const SharedFit& s, int a, int i) { return a * s.RS + i + (i >> 5); }

// Chain family F: 0 the rows (increasing in k), 1 the columns (decreasing in h), 2 the diagonal.
// Where a chain's list (and its blocks) start, and position p of it.
template <int F>
__device__ __forceinline__ int fit_base(const SharedFit& s, int ch) { return F == 0 ? ch * s.RS : F == 1 ? ch * s.MS : 0; }
template <int F>
__device__ __forceinline__ int fit_at(int p) { return F == 0 ? p + (p >> 5) : p; }
template <int F>
__device__ __forceinline__ int fit_len(const SharedFit& s, int ch) { return F == 0 ? s.rc[ch] : F == 1 ? s.cc[ch] : s.dc; }

// Pools a chain of len positions with values value(q, z, w) over a group of g lanes (this lane:
// ``part``; every lane of the warp calls it, a group without a chain with len = 0), weighted
// pool-adjacent-violators.  Position p's block entries are at at(p) of SM, SW and LK.
template <class Real, class AtF, class ValueF>
__device__ __forceinline__ void pool_chain(int part, int g, int len, Real* SM, Real* SW, unsigned short* LK, AtF at,
                                           ValueF value) {
    const int q0 = part * len / g, q1 = (part + 1) * len / g;
    // 1) this lane's run; the open block [bs, q] in registers
    {
        int bs = q0;
        Real ts = 0, tw = 0, nx = 0, nwt = 0;
        if (q0 < q1) value(q0, nx, nwt);
        for (int q = q0; q < q1; ++q) {
            Real w = nwt, sm = nx * nwt;
            if (q + 1 < q1) value(q + 1, nx, nwt);
            LK[at(q)] = 0;   // inside a block unless it comes to start or end one
            if (q > q0) {
                if (ts * w > sm * tw) {   // earlier mean > this mean
                    sm = ts + sm;
                    w = tw + w;
                    while (bs > q0) {
                        const int ps = LK[at(bs - 1)];
                        const Real psm = SM[at(ps)], psw = SW[at(ps)];
                        if (!(psm * w > sm * psw)) break;
                        sm = psm + sm;
                        w = psw + w;
                        bs = ps;
                        LK[at(ps)] = 0;   // open again
                    }
                } else {   // close the open block
                    SM[at(bs)] = ts;
                    SW[at(bs)] = tw;
                    LK[at(q - 1)] = static_cast<unsigned short>(bs);
                    LK[at(bs)] = static_cast<unsigned short>(q - 1);
                    bs = q;
                }
            }
            ts = sm;
            tw = w;
        }
        if (q0 < q1) {
            SM[at(bs)] = ts;
            SW[at(bs)] = tw;
            LK[at(q1 - 1)] = static_cast<unsigned short>(bs);
            LK[at(bs)] = static_cast<unsigned short>(q1 - 1);
        }
    }
    __syncwarp();
    // 2) join the runs of lanes [part - h, part) and [part, part + h)
    for (int h = 1; h < g; h <<= 1) {
        if ((part & (2 * h - 1)) == h) {
            const int b0 = (part - h) * len / g, b1 = (part + h) * len / g;
            if (b0 < q0 && q0 < b1) {
                int S = LK[at(q0 - 1)], E = LK[at(q0)];
                const Real lsm = SM[at(S)], lsw = SW[at(S)], rsm = SM[at(q0)], rsw = SW[at(q0)];
                if (lsm * rsw > rsm * lsw) {
                    Real sm = lsm + rsm, w = lsw + rsw;
                    LK[at(q0)] = static_cast<unsigned short>(S);   // no longer a start
                    for (;;) {
                        if (E + 1 < b1) {
                            const int s3 = E + 1, e3 = LK[at(s3)];
                            const Real xsm = SM[at(s3)], xsw = SW[at(s3)];
                            if (sm * xsw > xsm * w) {
                                sm += xsm;
                                w += xsw;
                                LK[at(s3)] = static_cast<unsigned short>(S);
                                E = e3;
                                continue;
                            }
                        }
                        if (S > b0) {
                            const int s0 = LK[at(S - 1)];
                            const Real xsm = SM[at(s0)], xsw = SW[at(s0)];
                            if (xsm * w > sm * xsw) {
                                sm += xsm;
                                w += xsw;
                                LK[at(S)] = static_cast<unsigned short>(s0);
                                S = s0;
                                continue;
                            }
                        }
                        break;
                    }
                    SM[at(S)] = sm;
                    SW[at(S)] = w;
                    LK[at(E)] = static_cast<unsigned short>(S);
                    LK[at(S)] = static_cast<unsigned short>(E);
                }
            }
        }
        __syncwarp();
    }
}

// Start of the block that covers this lane's first position when that is not a start itself
// (the last start of the group's lanes before it).
template <class AtF>
__device__ __forceinline__ int covering_start(int part, int g, int q0, int q1, const unsigned short* LK, AtF at) {
    int cover = -1;
    for (int q = q0; q < q1; ++q)
        if (LK[at(q)] >= q) cover = q;
    for (int o = 1; o < g; o <<= 1) {
        const int t = __shfl_up_sync(0xffffffffu, cover, o, g);
        if (part >= o) cover = max(cover, t);
    }
    return __shfl_up_sync(0xffffffffu, cover, 1, g);
}

// One Dykstra projection on family F; returns the thread's largest |change of x|.
template <int F>
__device__ float shared_phase(const SharedFit& s) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = s.T >> 5;
    const int nch = F == 0 ? s.m : F == 1 ? s.n : 1, most = F == 0 ? s.n : s.m;
    int g = 32;
    while (g > 1 && (g * nch > s.T || g / 2 >= most)) g >>= 1;
    const int per_warp = 32 / g, part = lane & (g - 1), sub = lane / g;
    const unsigned short* list0 = F == 0 ? s.rl : F == 1 ? s.cl : s.dl;
    float* pf = F == 0 ? s.P0 : F == 1 ? s.P1 : s.P2;
    float moved = 0.f;
    for (int c0 = warp * per_warp; c0 < nch; c0 += nw * per_warp) {
        const int ch = c0 + sub;
        const bool on = ch < nch;
        const int len = on ? fit_len<F>(s, ch) : 0;
        const int base = on ? fit_base<F>(s, ch) : 0;
        const unsigned short* list = list0 + base;
        float *SM = s.SM + base, *SW = s.SW + base;
        unsigned short* LK = s.LK + base;
        auto at = [](int p) { return fit_at<F>(p); };
        const int q0 = part * len / g, q1 = (part + 1) * len / g;
        // the dual of listed cell c at position q
        auto dual = [&](int c, int q) -> float& { return F == 2 ? pf[q] : pf[c]; };
        pool_chain(part, g, len, SM, SW, LK, at, [&](int q, float& z, float& w) {
            const int c = list[at(q)];
            z = s.X[c] + dual(c, q);
            w = s.W[c];
        });
        // every lane assigns its run
        const int cover = covering_start(part, g, q0, q1, LK, at);
        bool single = false;
        float val = 0.f;
        for (int q = q0; q < q1; ++q) {
            const int e = LK[at(q)];
            const bool start = e >= q;
            if (start || q == q0) {
                const int b = start ? q : cover;
                single = start && e == q;
                val = SM[at(b)] / SW[at(b)];
            }
            const int c = list[at(q)];
            float& pr = dual(c, q);
            const float old = s.X[c], z = old + pr;
            const float v = single ? z : val;
            pr = z - v;
            s.X[c] = v;
            moved = fmaxf(moved, fabsf(v - old));
        }
        __syncwarp();   // the next chains of this warp reuse nothing of these, but keep the lanes together
    }
    return moved;
}

// f(prev, c) for every pair of consecutive listed cells of family F.
template <int F, class EdgeF>
__device__ void shared_edges(const SharedFit& s, EdgeF f) {
    const int nch = F == 0 ? s.m : F == 1 ? s.n : 1, most = F == 0 ? s.n : s.m;
    const unsigned short* list0 = F == 0 ? s.rl : F == 1 ? s.cl : s.dl;
    for (int e = threadIdx.x; e < nch * most; e += s.T) {
        const int ch = e / most, q = e - ch * most;
        if (q < 1 || q >= fit_len<F>(s, ch)) continue;
        const unsigned short* list = list0 + fit_base<F>(s, ch);
        f(static_cast<int>(list[fit_at<F>(q - 1)]), static_cast<int>(list[fit_at<F>(q)]));
    }
}

// uf_find / uf_union on 16-bit parents.
__device__ __forceinline__ int uf_find16(volatile unsigned short* par, int x) {
    for (;;) {
        const int p = par[x];
        if (p == x) return x;
        const int gp = par[p];
        if (gp != p) par[x] = static_cast<unsigned short>(gp);
        x = p;
    }
}
__device__ __forceinline__ void uf_union16(unsigned short* par, int a, int b) {
    for (int guard = 0; guard < (1 << 22); ++guard) {
        a = uf_find16(par, a);
        b = uf_find16(par, b);
        if (a == b) return;
        if (a < b) {
            const int t = a;
            a = b;
            b = t;
        }
        const unsigned short me = static_cast<unsigned short>(a);
        if (atomicCAS(&par[a], me, static_cast<unsigned short>(b)) == me) return;
    }
}

// The whole fit once the group rows are known (v.rows, v.isrow; m >= 1).
__device__ void fit_in_shared(View& v, int n, int m, double tol, int max_sweeps, double* __restrict__ T_hat, char* smem,
                              float* red) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, T = blockDim.x, nw = T >> 5;
    const size_t nn = static_cast<size_t>(n) * n;
    const int32_t* cnt = v.cnt;
    SharedFit s;
    s.n = n;
    s.m = m;
    s.RS = fit_row_stride(n);
    s.MS = m | 1;
    s.T = T;
    const int C = static_cast<int>(fit_slots(n, m));
    char* at = smem;
    auto take = [&](size_t bytes) {
        char* r = at;
        at += bytes;
        return r;
    };
    const size_t N = static_cast<size_t>(n);
    s.mu = reinterpret_cast<double*>(take(N * 8));
    s.rows = reinterpret_cast<int*>(take(N * 4));
    s.isrow = reinterpret_cast<int*>(take(N * 4));
    s.P2 = reinterpret_cast<float*>(take(N * 4));
    s.rc = reinterpret_cast<unsigned short*>(take(N * 2));
    s.cc = reinterpret_cast<unsigned short*>(take(N * 2));
    s.dl = reinterpret_cast<unsigned short*>(take(N * 2));
    at = smem + fit_shared_fixed(n);
    const size_t C4 = static_cast<size_t>(C) * 4, C2 = static_cast<size_t>(C) * 2;
    s.P0 = reinterpret_cast<float*>(take(C4));   // P0 and P1 first: 8-byte words once the sweeps are over
    s.P1 = reinterpret_cast<float*>(take(C4));
    s.X = reinterpret_cast<float*>(take(C4));
    s.W = reinterpret_cast<float*>(take(C4));
    s.SM = reinterpret_cast<float*>(take(C4));
    s.SW = reinterpret_cast<float*>(take(C4));
    s.LK = reinterpret_cast<unsigned short*>(take(C2));
    s.par = reinterpret_cast<unsigned short*>(take(C2));
    s.rl = reinterpret_cast<unsigned short*>(take(C2));
    s.cl = reinterpret_cast<unsigned short*>(take(C2));
    s.dc = m;   // every group row's diagonal cell is observed
    for (int i = tid; i < n; i += T) {
        s.isrow[i] = v.isrow[i];
        if (i < m) s.rows[i] = v.rows[i];
    }
    // pooled column means (exact sums, fp64) over the rows that have samples (listed in P2)
    int* seen_rows = reinterpret_cast<int*>(s.P2);
    for (int h = warp; h < n; h += nw) {
        int any = 0;
#pragma unroll 8
        for (int i = lane; i < n; i += 32) any |= cnt[static_cast<size_t>(h) * n + i];
        any = __any_sync(0xffffffffu, any != 0);
        if (lane == 0) s.rc[h] = static_cast<unsigned short>(any);
    }
    __syncthreads();
    int nseen = 0;
    if (warp == 0) {
        for (int h0 = 0; h0 < n; h0 += 32) {
            const bool on = h0 + lane < n && s.rc[h0 + lane] != 0;
            const unsigned bal = __ballot_sync(0xffffffffu, on);
            if (on) seen_rows[nseen + __popc(bal & ((1u << lane) - 1u))] = h0 + lane;
            nseen += __popc(bal);
        }
        if (lane == 0) s.cc[0] = static_cast<unsigned short>(nseen);
    }
    __syncthreads();
    nseen = s.cc[0];
    bool empty = false;
    for (int i = tid; i < n; i += T) {
        unsigned long long sm = 0;
        long long c = 0;
#pragma unroll 8
        for (int q = 0; q < nseen; ++q) {
            const size_t g = static_cast<size_t>(seen_rows[q]) * n + i;
            sm += v.sum[g];
            c += cnt[g];
        }
        s.mu[i] = c > 0 ? (static_cast<double>(sm) * kUnit) / static_cast<double>(c) : CUDART_NAN;
        empty |= c == 0;
    }
    if (__syncthreads_or(empty) && tid == 0) {   // empty columns: the nearest earlier column, else the nearest later
        int first = -1;
        for (int i = 0; i < n; ++i) {
            if (isnan(s.mu[i])) {
                if (i > 0) s.mu[i] = s.mu[i - 1];
            } else if (first < 0) {
                first = i;
            }
        }
        for (int i = 0; i < first; ++i) s.mu[i] = s.mu[first];
    }
    __syncthreads();   // seen_rows' memory is P2's from here
    // targets, weights, warm start, as in the state-buffer form
    float* lam0 = v.lam;
    float* lam1 = v.lam + nn;
    float* lam2 = v.lam + 2 * nn;
    const int cells = m * n;
    float ymax = 0.f;
    for (int q = tid; q < cells; q += T) {
        const int a = q / n, i = q - a * n;
        const int c = fit_cell(s, a, i);
        const size_t g = static_cast<size_t>(s.rows[a] - 1) * n + i;
        const int k = cnt[g];
        s.par[c] = static_cast<unsigned short>(c);
        if (i == s.rows[a] - 1) s.P2[a] = 0.f;
        if (k == 0) {
            s.W[c] = 0.f;
            continue;
        }
        const float w = static_cast<float>(k);
        const float y = static_cast<float>((static_cast<double>(v.sum[g]) * kUnit) / static_cast<double>(k));
        const float p0 = lam0[g] / w, p1 = lam1[g] / w, p2 = lam2[g] / w;
        s.W[c] = w;
        s.P0[c] = p0;
        s.P1[c] = p1;
        if (i == s.rows[a] - 1) s.P2[a] = p2;
        s.X[c] = y - ((p0 + p1) + p2);
        ymax = fmaxf(ymax, fabsf(y));
    }
    const float tol_abs = fmaxf(static_cast<float>(tol), kMinTol) * block_max(ymax, red);   // (its barriers end the set-up)
    // the observed cells of each chain
    for (int a = warp; a < m; a += nw) {
        int count = 0;
        for (int i0 = 0; i0 < n; i0 += 32) {
            const int i = i0 + lane;
            const bool seen = i < n && s.W[fit_cell(s, a, i)] > 0.f;
            const unsigned bal = __ballot_sync(0xffffffffu, seen);
            if (seen)
                s.rl[fit_base<0>(s, a) + fit_at<0>(count + __popc(bal & ((1u << lane) - 1u)))] =
                    static_cast<unsigned short>(fit_cell(s, a, i));
            count += __popc(bal);
        }
        if (lane == 0) {
            s.rc[a] = static_cast<unsigned short>(count);
            s.dl[a] = static_cast<unsigned short>(fit_cell(s, a, s.rows[a] - 1));
        }
    }
    for (int i = tid; i < n; i += T) {
        int count = 0;
        for (int a = m - 1; a >= 0; --a) {
            const int c = fit_cell(s, a, i);
            if (s.W[c] > 0.f) s.cl[fit_base<1>(s, i) + count++] = static_cast<unsigned short>(c);
        }
        s.cc[i] = static_cast<unsigned short>(count);
    }
    __syncthreads();

    int sweeps = 0;
    bool converged = false;
    while (sweeps < max_sweeps) {
        ++sweeps;
        float moved = shared_phase<0>(s);
        __syncthreads();
        moved = fmaxf(moved, shared_phase<1>(s));
        __syncthreads();
        moved = fmaxf(moved, shared_phase<2>(s));
        if (block_max(moved, red) * 3.f <= tol_abs) {
            converged = true;
            break;
        }
    }
    __syncthreads();
    if (converged) {   // one more sweep, recording the blocks (record_sweep)
        auto join = [&](int a, int b) {
            if (s.X[a] == s.X[b]) uf_union16(s.par, a, b);
        };
        shared_phase<0>(s);
        __syncthreads();
        shared_edges<0>(s, join);
        __syncthreads();
        shared_phase<1>(s);
        __syncthreads();
        shared_edges<1>(s, join);
        __syncthreads();
        shared_phase<2>(s);
        __syncthreads();
        shared_edges<2>(s, join);
        __syncthreads();
    }
    // keep the dual variables for the next fit; their shared memory is free after that
    for (int q = tid; q < cells; q += T) {
        const int a = q / n, i = q - a * n;
        const int c = fit_cell(s, a, i);
        const float w = s.W[c];
        if (!(w > 0.f)) continue;
        const size_t g = static_cast<size_t>(s.rows[a] - 1) * n + i;
        lam0[g] = s.P0[c] * w;
        lam1[g] = s.P1[c] * w;
        if (i == s.rows[a] - 1) lam2[g] = s.P2[a] * w;
        v.x[g] = s.X[c];
    }
    __syncthreads();
    // exact block means (fp64 from the int64 cell sums)
    unsigned long long* csum = reinterpret_cast<unsigned long long*>(s.P0);   // over P0 and P1
    int* ccnt = reinterpret_cast<int*>(s.SM);
    int* root = reinterpret_cast<int*>(s.SW);
    bool polished = false;
    if (converged) {
        auto greater = [&](int a, int b) {
            const int ra = root[a], rb = root[b];
            if (ra == rb) return false;
            const unsigned long long sa = csum[ra], sb = csum[rb];
            const unsigned long long ca = static_cast<unsigned long long>(ccnt[ra]);
            const unsigned long long cb = static_cast<unsigned long long>(ccnt[rb]);
            const unsigned long long hi1 = __umul64hi(sa, cb), lo1 = sa * cb;
            const unsigned long long hi2 = __umul64hi(sb, ca), lo2 = sb * ca;
            return hi1 > hi2 || (hi1 == hi2 && lo1 > lo2);
        };
        int merged;
        auto fix = [&](int a, int b) {   // pairs that break the order join one block
            if (greater(a, b)) {
                uf_union16(s.par, a, b);
                merged = 1;
            }
        };
        const int per = (cells + T - 1) / T;   // each thread owns a contiguous run of cells
        const int r0 = tid * per < cells ? tid * per : cells, r1 = r0 + per < cells ? r0 + per : cells;
        for (int round = 0; round < kFixRounds; ++round) {
            for (int jump = 0; jump < 32; ++jump) {   // flatten the trees by pointer jumping
                bool moved = false;
                for (int q = r0; q < r1; ++q) {
                    const int a = q / n, c = fit_cell(s, a, q - a * n);
                    if (!(s.W[c] > 0.f)) continue;
                    volatile unsigned short* par = s.par;
                    const int pc = par[c], gp = par[pc];
                    if (gp != pc) {
                        par[c] = static_cast<unsigned short>(gp);
                        moved = true;
                    }
                }
                if (!__syncthreads_or(moved)) break;
            }
            for (int q = r0; q < r1; ++q) {
                const int a = q / n, c = fit_cell(s, a, q - a * n);
                if (!(s.W[c] > 0.f)) continue;
                root[c] = uf_find16(s.par, c);
                csum[c] = 0ull;
                ccnt[c] = 0;
            }
            __syncthreads();
            int cur = -1, cn = 0;   // exact sums per block: a run of cells with the same root adds once
            unsigned long long sm = 0ull;
            for (int q = r0; q < r1; ++q) {
                const int a = q / n, i = q - a * n, c = fit_cell(s, a, i);
                if (!(s.W[c] > 0.f)) continue;
                const int r = root[c];
                if (r != cur) {
                    if (cur >= 0) {
                        atomicAdd(csum + cur, sm);
                        atomicAdd(ccnt + cur, cn);
                    }
                    cur = r;
                    sm = 0ull;
                    cn = 0;
                }
                const size_t g = static_cast<size_t>(s.rows[a] - 1) * n + i;
                sm += v.sum[g];
                cn += cnt[g];
            }
            if (cur >= 0) {
                atomicAdd(csum + cur, sm);
                atomicAdd(ccnt + cur, cn);
            }
            __syncthreads();
            merged = 0;
            shared_edges<0>(s, fix);
            shared_edges<1>(s, fix);
            shared_edges<2>(s, fix);
            if (!__syncthreads_or(merged)) {
                polished = true;
                break;
            }
        }
        if (polished) {   // each cell's exact block mean (fp64), and its fp32 copy
            for (int q = tid; q < cells; q += T) {
                const int a = q / n, i = q - a * n, c = fit_cell(s, a, i);
                if (!(s.W[c] > 0.f)) continue;
                const int r = root[c];
                const double mc = (static_cast<double>(csum[r]) * kUnit) / static_cast<double>(ccnt[r]);
                const size_t g = static_cast<size_t>(s.rows[a] - 1) * n + i;
                v.xd[g] = mc;
                v.x[g] = static_cast<float>(mc);
            }
        }
    }
    __syncthreads();
    auto fitted = [&](size_t g) { return polished ? v.xd[g] : static_cast<double>(v.x[g]); };
    // the observed ranks around each rank of a row: the last one <= i (plus 1, 0: none), the
    // first one >= i (n: none)
    unsigned short* before = reinterpret_cast<unsigned short*>(s.SM);
    unsigned short* after = before + C;
    for (int a = warp; a < m; a += nw) {
        int carry = 0;
        for (int i0 = 0; i0 < n; i0 += 32) {
            const int i = i0 + lane;
            const unsigned seen = __ballot_sync(0xffffffffu, i < n && s.W[fit_cell(s, a, i < n ? i : 0)] > 0.f);
            const unsigned upto = seen & (0xffffffffu >> (31 - lane));
            if (i < n) before[fit_cell(s, a, i)] = static_cast<unsigned short>(upto ? i0 + 32 - __clz(upto) : carry);
            if (seen) carry = i0 + 32 - __clz(seen);
        }
        carry = n;
        for (int i0 = (n - 1) / 32 * 32; i0 >= 0; i0 -= 32) {
            const int i = i0 + lane;
            const unsigned seen = __ballot_sync(0xffffffffu, i < n && s.W[fit_cell(s, a, i < n ? i : 0)] > 0.f);
            const unsigned from = seen & (0xffffffffu << lane);
            if (i < n) after[fit_cell(s, a, i)] = static_cast<unsigned short>(from ? i0 + __ffs(from) - 1 : carry);
            if (seen) carry = i0 + __ffs(seen) - 1;
        }
    }
    // diagonal cells outside the group: pooled column means, nondecreasing (PAVA in fp64, unit
    // weights), by one warp, over the block sums' and dual variables' memory (one thread took 140
    // of the 250 us outside the sweeps at n = 256: a dependent fp64 operation is slow here)
    if (warp == 0) {
        double* bs = reinterpret_cast<double*>(s.P0);   // n - m entries each: see fit_shared_fits
        double* bw = bs + (n - m);
        unsigned short *LK = s.LK, *free_k = s.par;
        int len = 0;
        for (int k0 = 0; k0 < n; k0 += 32) {
            const bool on = k0 + lane < n && s.isrow[k0 + lane] < 0;
            const unsigned bal = __ballot_sync(0xffffffffu, on);
            if (on) free_k[len + __popc(bal & ((1u << lane) - 1u))] = static_cast<unsigned short>(k0 + lane);
            len += __popc(bal);
        }
        __syncwarp();
        auto at = [](int p) { return p; };
        pool_chain(lane, 32, len, bs, bw, LK, at, [&](int q, double& z, double& w) {
            z = s.mu[free_k[q]];
            w = 1.0;
        });
        const int q0 = lane * len / 32, q1 = (lane + 1) * len / 32;
        const int cover = covering_start(lane, 32, q0, q1, LK, at);
        int b = -1;
        double val = 0.0;
        for (int q = q0; q < q1; ++q) {
            const int e = LK[q];
            const bool start = e >= q;
            if (start || q == q0) {
                b = start ? q : cover;
                val = bs[b] / bw[b];
            }
            if (!(start && e == q)) s.mu[free_k[q]] = val;   // a block of one keeps its mean as it is
        }
    }
    if (tid == 0) {
        v.hdr->sweeps = sweeps;
        if (!converged) v.hdr->flags |= DBW_PSW_NOT_CONVERGED;
        if (converged && !polished) v.hdr->flags |= DBW_PSW_UNPOLISHED;
    }
    __syncthreads();
    // ... clipped to the bounds the fitted cells place on them: the largest of j <= min(h, k) is
    // at the last observed one, the smallest of j >= max(h, k) at the first observed one
    for (int k = tid; k < n; k += T) {
        const int kk = k + 1;
        if (s.isrow[k] >= 0) {
            T_hat[k] = fitted(static_cast<size_t>(k) * (n + 1));
        } else {
            double lo = -CUDART_INF, hi = CUDART_INF;
#pragma unroll 4
            for (int a = 0; a < m; ++a) {
                const int h = s.rows[a];
                const size_t base = static_cast<size_t>(h - 1) * n;
                const int below = before[fit_cell(s, a, min(h, kk) - 1)];
                const int above = after[fit_cell(s, a, max(h, kk) - 1)];
                if (below > 0) lo = fmax(lo, fitted(base + below - 1));
                if (above < n) hi = fmin(hi, fitted(base + above));
            }
            T_hat[k] = fmin(fmax(s.mu[k], lo), hi);
        }
    }
}

constexpr size_t kFitSharedMax = 231000;   // dynamic shared memory of the fit (227 KB less its static part)
// Whether the m x n table fits; the PAVA of the n - m free diagonal cells lies over P0 .. P1
// (16 bytes each), LK and par (2 bytes each).
__device__ __forceinline__ bool fit_shared_fits(int n, int m, size_t bytes) {
    const size_t C = fit_slots(n, m), free_cells = static_cast<size_t>(n - m);
    return fit_shared_bytes(n, m) <= bytes && C < 65536 && free_cells * 16 <= C * 8 && free_cells <= C;
}

// Group rows (diagonal cell has samples), in increasing h: v.rows, v.isrow; returns their
// number.  The whole block calls it; ends in a barrier.
__device__ int group_rows(View& v, int n, int* warp_tot) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    int m = 0;
    for (int h0 = 0; h0 < n; h0 += blockDim.x) {
        const int h = h0 + tid;
        const bool has = h < n && v.cnt[static_cast<size_t>(h) * (n + 1)] > 0;
        const unsigned bal = __ballot_sync(0xffffffffu, has);
        if (lane == 0) warp_tot[warp] = __popc(bal);
        __syncthreads();
        int pos = m + __popc(bal & ((1u << lane) - 1u));
        for (int q = 0; q < static_cast<int>(blockDim.x >> 5); ++q) {
            if (q < warp) pos += warp_tot[q];
            m += warp_tot[q];
        }
        if (h < n) {
            v.isrow[h] = has ? pos : -1;
            if (has) v.rows[pos] = h + 1;
        }
        __syncthreads();
    }
    return m;
}

// The fit of a table that fits in shared memory; leaves the others to psw_estimate_kernel,
// the next launch, which sees the same counts and so decides the same way.
__global__ void __launch_bounds__(1024, 1) psw_fit_shared_kernel(char* base, Layout L, int n, double tol,
                                                                  int max_sweeps, double* __restrict__ T_hat,
                                                                  size_t shared_bytes) {
    grid_begin();
    extern __shared__ __align__(16) char fit_smem[];
    __shared__ int warp_tot[32];
    __shared__ float red[32];
    View v = view(base, L);
    const int m = group_rows(v, n, warp_tot);
    if (m == 0) {
        for (int k = threadIdx.x; k < n; k += blockDim.x) T_hat[k] = CUDART_NAN;
        if (threadIdx.x == 0) v.hdr->sweeps = 0;
        return;
    }
    if (fit_shared_fits(n, m, shared_bytes)) fit_in_shared(v, n, m, tol, max_sweeps, T_hat, fit_smem, red);
}

// The fit of Eq. (17) on the state buffer, one CTA of fit_threads(n) threads.
template <int MAXT>
__global__ void __launch_bounds__(MAXT, 1) psw_estimate_kernel(char* base, Layout L, int n, double tol,
                                                                int max_sweeps, double* __restrict__ T_hat,
                                                                size_t shared_bytes) {
    grid_begin();
    __shared__ int warp_tot[32];
    __shared__ float red[32];
    __shared__ int fix_s, polished_s, jump_s;
    View v = view(base, L);
    const int tid = threadIdx.x;
    const int T = blockDim.x;
    const size_t nn = static_cast<size_t>(n) * n;
    float* lam0 = v.lam;
    float* lam1 = v.lam + nn;
    float* lam2 = v.lam + 2 * nn;
    const int32_t* cnt = v.cnt;

    const int m = group_rows(v, n, warp_tot);
    if (m == 0 || fit_shared_fits(n, m, shared_bytes)) return;   // psw_fit_shared_kernel did it
    // pooled column means (exact sums, fp64)
    if (tid < n) {
        unsigned long long sm = 0;
        long long c = 0;
        for (int h = 0; h < n; ++h) {
            sm += v.sum[static_cast<size_t>(h) * n + tid];
            c += cnt[static_cast<size_t>(h) * n + tid];
        }
        v.mu[tid] = c > 0 ? (static_cast<double>(sm) * kUnit) / static_cast<double>(c) : CUDART_NAN;
    }
    __syncthreads();
    if (tid == 0) {   // empty columns: the nearest earlier column with samples, else the nearest later
        int first = -1;
        for (int i = 0; i < n; ++i) {
            if (isnan(v.mu[i])) {
                if (i > 0) v.mu[i] = v.mu[i - 1];
            } else if (first < 0) {
                first = i;
            }
        }
        for (int i = 0; i < first; ++i) v.mu[i] = v.mu[first];
    }
    __syncthreads();

    const int32_t* rows = v.rows;
    const size_t cells = static_cast<size_t>(m) * n;
    // targets (cell means), weights (counts), warm start: x = y - sum_f lambda_f / w
    float ymax = 0.f;
    for (size_t q = tid; q < cells; q += T) {
        const size_t c = static_cast<size_t>(rows[q / n] - 1) * n + q % n;
        const int k = cnt[c];
        if (k == 0) {
            v.w[c] = 0.f;
            continue;
        }
        const float w = static_cast<float>(k);
        const float y = static_cast<float>((static_cast<double>(v.sum[c]) * kUnit) / static_cast<double>(k));
        v.w[c] = w;
        const float p0 = lam0[c] / w, p1 = lam1[c] / w, p2 = lam2[c] / w;
        lam0[c] = p0;
        lam1[c] = p1;
        lam2[c] = p2;
        v.x[c] = y - ((p0 + p1) + p2);
        ymax = fmaxf(ymax, fabsf(y));
    }
    const float tol_abs = fmaxf(static_cast<float>(tol), kMinTol) * block_max(ymax, red);

    int sweeps = 0;
    bool converged = false;
    auto idx = [=](int a, int i) { return (rows[a] - 1) * n + i; };
    sweeps = dykstra_sweeps(v.x, lam0, lam1, lam2, v.w, idx, rows, m, n, v.bm, v.bw, v.bl, v.bp, v.ab, v.nbk, v.mv, T,
                            tol_abs, max_sweeps, red, &converged);
    __syncthreads();

    // exact block means (fp64 from the int64 cell sums) once the sweeps have converged
    int32_t* par = v.par;
    int32_t* root = v.root;
    unsigned long long* csum = v.csum;
    int32_t* ccnt = v.ccnt;
    if (tid == 0) polished_s = 0;
    if (converged) {
        for (size_t q = tid; q < cells; q += T) {
            const int c = static_cast<int>(static_cast<size_t>(rows[q / n] - 1) * n + q % n);
            par[c] = c;
        }
        __syncthreads();
        record_sweep(v.x, lam0, lam1, lam2, v.w, idx, rows, m, n, v.bm, v.bw, v.bl, v.bp, v.ab, v.nbk, v.mv, T, par);
        auto rowf = [=](int a, int q) { return idx(a, q); };
        auto colf = [=](int i, int q) { return idx(m - 1 - q, i); };
        auto diagf = [=](int, int q) { return idx(q, rows[q] - 1); };
        auto mean = [=](int c) {
            const int r = root[c];
            return (static_cast<double>(csum[r]) * kUnit) / static_cast<double>(ccnt[r]);
        };
        // mean of a's block > mean of b's block, exactly: sum_a cnt_b > sum_b cnt_a in
        // 128-bit integers (the sums are nonnegative fixed point)
        auto greater = [=](int a, int b) {
            const int ra = root[a], rb = root[b];
            if (ra == rb) return false;
            const unsigned long long sa = csum[ra], sb = csum[rb];
            const unsigned long long ca = static_cast<unsigned long long>(ccnt[ra]);
            const unsigned long long cb = static_cast<unsigned long long>(ccnt[rb]);
            const unsigned long long hi1 = __umul64hi(sa, cb), lo1 = sa * cb;
            const unsigned long long hi2 = __umul64hi(sb, ca), lo2 = sb * ca;
            return hi1 > hi2 || (hi1 == hi2 && lo1 > lo2);
        };
        // pairs that break the order join one block; *fixp notes that a round merged
        int* fixp = &fix_s;
        auto fix = [=](int a, int b) {
            if (greater(a, b)) {
                uf_union(par, a, b);
                *fixp = 1;
            }
        };
        // each thread owns a contiguous run of cells (row-major: neighbours mostly share a block)
        const size_t per = (cells + T - 1) / T;
        const size_t q0 = tid * per < cells ? tid * per : cells;
        const size_t q1 = q0 + per < cells ? q0 + per : cells;
        auto cell_of = [=](size_t q) { return static_cast<int>(static_cast<size_t>(rows[q / n] - 1) * n + q % n); };
        for (int round = 0; round < kFixRounds; ++round) {
            // flatten the trees: pointer jumping (parents stay ancestors, so concurrent
            // updates only shorten the paths), then each cell's root
            for (int jump = 0; jump < 32; ++jump) {
                if (tid == 0) jump_s = 0;
                __syncthreads();
                bool moved = false;
                for (size_t q = q0; q < q1; ++q) {
                    const int c = cell_of(q);
                    if (cnt[c] == 0) continue;
                    const int pc = par[c];
                    const int gp = par[pc];
                    if (gp != pc) {
                        par[c] = gp;
                        moved = true;
                    }
                }
                if (moved) jump_s = 1;
                __syncthreads();
                const int more = jump_s;
                __syncthreads();
                if (!more) break;
            }
            for (size_t q = q0; q < q1; ++q) {
                const int c = cell_of(q);
                if (cnt[c] == 0) continue;
                root[c] = uf_find(par, c);
                csum[c] = 0ull;
                ccnt[c] = 0;
            }
            if (tid == 0) fix_s = 0;
            __syncthreads();
            {   // exact sums per block: a run of cells with the same root adds once
                int cur = -1, cn = 0;
                unsigned long long sm = 0ull;
                for (size_t q = q0; q < q1; ++q) {
                    const int c = cell_of(q);
                    if (cnt[c] == 0) continue;
                    const int r = root[c];
                    if (r != cur) {
                        if (cur >= 0) {
                            atomicAdd(csum + cur, sm);
                            atomicAdd(ccnt + cur, cn);
                        }
                        cur = r;
                        sm = 0ull;
                        cn = 0;
                    }
                    sm += v.sum[c];
                    cn += cnt[c];
                }
                if (cur >= 0) {
                    atomicAdd(csum + cur, sm);
                    atomicAdd(ccnt + cur, cn);
                }
            }
            __syncthreads();
            for_chain_edges(v.w, rowf, m, n, T, fix);
            for_chain_edges(v.w, colf, n, m, T, fix);
            for_chain_edges(v.w, diagf, 1, m, T, fix);
            __syncthreads();
            const int again = fix_s;
            __syncthreads();
            if (!again) {
                if (tid == 0) polished_s = 1;
                break;
            }
        }
        __syncthreads();
        if (polished_s) {   // each cell's exact block mean (fp64), and its fp32 copy
            for (size_t q = tid; q < cells; q += T) {
                const int c = static_cast<int>(static_cast<size_t>(rows[q / n] - 1) * n + q % n);
                if (cnt[c] == 0) continue;
                const double mc = mean(c);
                v.xd[c] = mc;
                v.x[c] = static_cast<float>(mc);
            }
        }
    }
    __syncthreads();
    const bool polished = polished_s != 0;
    // value of a fitted group cell: its exact block mean, else the fp32 fit
    auto fitted = [=](int c) { return polished ? v.xd[c] : static_cast<double>(v.x[c]); };
    // keep the dual variables for the next fit
    for (size_t q = tid; q < cells; q += T) {
        const size_t c = static_cast<size_t>(rows[q / n] - 1) * n + q % n;
        if (cnt[c] == 0) continue;
        lam0[c] *= v.w[c];
        lam1[c] *= v.w[c];
        lam2[c] *= v.w[c];
    }
    // diagonal cells outside the group: pooled column means, nondecreasing (PAVA in
    // fp64, unit weights), clipped to the bounds the fitted cells place on them
    if (tid == 0) {
        double* bs = v.fd;
        double* bw = v.fd + n;
        int* bl = v.bl;
        int nb = 0;
        for (int k = 0; k < n; ++k) {
            if (v.isrow[k] >= 0) continue;
            double sm = v.mu[k], ww = 1.0;
            int l = 1;
            while (nb > 0 && bs[nb - 1] * ww > sm * bw[nb - 1]) {
                sm = bs[nb - 1] + sm;
                ww = bw[nb - 1] + ww;
                l += bl[nb - 1];
                --nb;
            }
            bs[nb] = sm;
            bw[nb] = ww;
            bl[nb] = l;
            ++nb;
        }
        int b = 0, left = nb > 0 ? bl[0] : 0;
        for (int k = 0; k < n && b < nb; ++k) {
            if (v.isrow[k] >= 0) continue;
            T_hat[k] = bl[b] == 1 ? v.mu[k] : bs[b] / bw[b];
            if (--left == 0 && ++b < nb) left = bl[b];
        }
        v.hdr->sweeps = sweeps;
        if (!converged) v.hdr->flags |= DBW_PSW_NOT_CONVERGED;
        if (converged && !polished) v.hdr->flags |= DBW_PSW_UNPOLISHED;
    }
    __syncthreads();
    for (int k = tid; k < n; k += T) {
        const int kk = k + 1;
        if (v.isrow[k] >= 0) {
            T_hat[k] = fitted(k * (n + 1));
        } else {
            // group rows are nondecreasing along their observed cells: the largest of
            // j <= min(h, k) is at the last observed j <= min(h, k), the smallest of
            // j >= max(h, k) at the first observed j >= max(h, k)
            double lo = -CUDART_INF, hi = CUDART_INF;
            for (int a = 0; a < m; ++a) {
                const int h = rows[a];
                const int base_c = (h - 1) * n;
                for (int j = min(h, kk); j >= 1; --j)
                    if (cnt[base_c + j - 1] > 0) {
                        lo = fmax(lo, fitted(base_c + j - 1));
                        break;
                    }
                for (int j = max(h, kk); j <= n; ++j)
                    if (cnt[base_c + j - 1] > 0) {
                        hi = fmin(hi, fitted(base_c + j - 1));
                        break;
                    }
            }
            T_hat[k] = fmin(fmax(T_hat[k], lo), hi);
        }
    }
}

}  // namespace

size_t psw_bytes(int n) { return layout(n).bytes; }

cudaError_t launch_psw_init(void* psw, int n, cudaStream_t st) {
    const Layout L = layout(n);
    cudaError_t e = cudaMemsetAsync(psw, 0, L.bytes, st);
    if (e != cudaSuccess) return e;
    launch(psw_init_kernel, 1, 32, 0, st, static_cast<char*>(psw), L, n);
    return cudaGetLastError();
}

cudaError_t launch_psw_arrivals(const void* psw, int n, const double* omega, double* e, cudaStream_t st) {
    launch(psw_arrivals_kernel, (n + 255) / 256, 256, 0, st, static_cast<const char*>(psw), layout(n), n, omega, e);
    return cudaGetLastError();
}

cudaError_t launch_psw_record(void* psw, int n, const int32_t* order, const double* tsorted, const int32_t* k,
                              cudaStream_t st) {
    launch(psw_record_kernel, 1, kThreads, 0, st, static_cast<char*>(psw), layout(n), n, order, tsorted, k);
    return cudaGetLastError();
}

cudaError_t launch_psw_estimate(void* psw, int n, double tol, int max_sweeps, double* T_hat, cudaStream_t st) {
    const Layout L = layout(n);
    char* base = static_cast<char*>(psw);
    // room for as many group rows as the table can have, within what a CTA can take; the opt-in,
    // which the host's threads share, is the same for every n
    const size_t all = fit_shared_bytes(n, n), smem = all < kFitSharedMax ? all : kFitSharedMax;
    cudaError_t e = cudaFuncSetAttribute(psw_fit_shared_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kFitSharedMax);
    if (e == cudaSuccess) e = launch(psw_fit_shared_kernel, 1, fit_shared_threads(n), smem, st, base, L, n, tol, max_sweeps, T_hat, smem);
    if (e != cudaSuccess) return e;
    const int T = fit_threads(n);
    auto kern = T <= 512 ? psw_estimate_kernel<512> : psw_estimate_kernel<kThreads>;   // fewer threads leave each more registers
    // not early: its tables live in L1, and a CTA set up beside other kernels finds its SM's L1
    // sized for those (n = 256: 5.0 ms, early 7.3)
    return launch_when(false, kern, 1, T, 0, st, base, L, n, tol, max_sweeps, T_hat, smem);
}

}  // namespace dbw
