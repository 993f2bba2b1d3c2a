// bf16 GEMM on the 5th-generation tensor cores of sm_103a (tcgen05), written
// with inline PTX: TMA (cp.async.bulk.tensor) loads into a ring of shared
// memory stages guarded by mbarriers, one thread issuing tcgen05.mma into a
// TMEM accumulator, and four epilogue warps reading TMEM with tcgen05.ld.
//
//   C[M, N] = sum_k A(m, k) * B(n, k)      (bf16 operands, fp32 accumulation)
//
// Operands stay in the row-major layout their producer wrote.  One whose rows run along
// K (activations and dZ as forward operands, W in the forward pass) is staged K-major:
// 64-element K slices of the tile's rows.  One whose rows run along M or N (dZ and the
// activations in the weight gradients, W in the input gradient) is staged MN-major:
// groups of 64 columns, each group one row per K index; the UMMA descriptors say which
// (tc_ptx.cuh).  Both use 128-byte rows with the 128-byte swizzle.
//
// CTA = 6 warps:  warp 0  TMA producer (one lane) and TMEM owner
//                 warp 1  MMA issuer (one lane)
//                 warps 2-5  epilogue: warp w reads TMEM lanes 32*(w%4) .. +31,
//                            i.e. rows m0 + 32*(w%4) + lane of the 128-row tile.
//
// Every wait on an mbarrier is bounded (2 s of %globaltimer).  A wait that runs
// out sets bit 0 of *status, the producer drains the TMA loads it still has in
// flight (again bounded), TMEM is freed and the CTA returns; the results of that
// launch are then undefined, never a fault or a hang.
#include <cuda.h>

#include <atomic>
#include <mutex>

#include "gemm_tc.cuh"
#include "profile.cuh"
#include "tc_ptx.cuh"

namespace dbw {

namespace {

using namespace tcx;

constexpr int BM = 128;
constexpr int kThreads = 192;

// Whether the rows of operand A / B of a GEMM kind run along M / N (MN-major staging).
__host__ __device__ constexpr bool a_mn(int kind) { return kind == TC_GBAR || kind == TC_DW; }
__host__ __device__ constexpr bool b_mn(int kind) { return kind == TC_GBAR || kind == TC_DW || kind == TC_DX; }

// Descriptor of K step kk (16 elements) of an operand tile staged at ``base`` in BK-deep stages.
template <bool MN, int BK>
__device__ __forceinline__ uint64_t operand_desc(uint32_t base, int kk) {
    return MN ? smem_desc_mn(base + kk * 2048, BK * 128) : smem_desc(base + kk * 32, 128);
}

// ------------------------------------------------------------------ epilogues
// One thread: row ``row`` of the tile, 32 columns starting at ``nb`` (logits and the
// one-CTA-per-tile weight-gradient kernel).
template <int KIND>
__device__ __forceinline__ void epilogue_chunk(const TcEpi& e, int z, int row, int nb, int M, int N,
                                               const uint32_t (&r)[32]) {
    if (row >= M) return;
    const bool full = nb + 32 <= N;
    if constexpr (KIND == TC_LOGITS) {
        float* op = e.outF + static_cast<int64_t>(row) * e.ldF + nb;
        if (full && ((reinterpret_cast<uintptr_t>(op) & 15u) == 0)) {
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                float4 v;
                v.x = u2f(r[4 * q + 0]) + __ldg(e.bias + nb + 4 * q + 0);
                v.y = u2f(r[4 * q + 1]) + __ldg(e.bias + nb + 4 * q + 1);
                v.z = u2f(r[4 * q + 2]) + __ldg(e.bias + nb + 4 * q + 2);
                v.w = u2f(r[4 * q + 3]) + __ldg(e.bias + nb + 4 * q + 3);
                *reinterpret_cast<float4*>(op + 4 * q) = v;
            }
        } else {
#pragma unroll
            for (int j = 0; j < 32; ++j)
                if (nb + j < N) op[j] = u2f(r[j]) + __ldg(e.bias + nb + j);
        }
    } else {   // TC_DW: element (m, n) -> G[z*ldG + off + m*ldrow + n]
        static_assert(KIND == TC_DW, "epilogue_chunk serves TC_LOGITS and TC_DW");
        float* op = e.G + static_cast<int64_t>(z) * e.ldG + e.off + static_cast<int64_t>(row) * e.ldrow + nb;
#pragma unroll
        for (int j = 0; j < 32; ++j)
            if (nb + j < N) __stcs(op + j, u2f(r[j]));
    }
}

// ------------------------------------------------------------------ epilogues of the pair kernel
// One thread owns one output row and 128 columns of a tile (four 32-column chunks
// read from TMEM at ``taddr``).  GBAR's loads of w for the SGD step are issued one
// chunk ahead, so that their latency overlaps the previous chunk's work.

// bf16 activation chunk (32 columns of row ``row``) -> out.  ``wide``: rows of out start on 32
// bytes, so that each store writes a whole sector per lane.
__device__ __forceinline__ void store_act_chunk(const TcEpi& e, int row, int nb, int N, const float (&x)[32],
                                                bool wide) {
    __nv_bfloat16* op = e.out + static_cast<int64_t>(row) * e.ldo + nb;
    if (nb + 32 <= N && wide) {
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            uint32_t w[8];
#pragma unroll
            for (int j = 0; j < 8; ++j) w[j] = pack_bf16(x[16 * q + 2 * j], x[16 * q + 2 * j + 1]);
            store_256(op + 16 * q, w);
        }
    } else if (nb + 32 <= N && ((reinterpret_cast<uintptr_t>(op) & 15u) == 0)) {
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            uint4 w;
            w.x = pack_bf16(x[8 * q + 0], x[8 * q + 1]);
            w.y = pack_bf16(x[8 * q + 2], x[8 * q + 3]);
            w.z = pack_bf16(x[8 * q + 4], x[8 * q + 5]);
            w.w = pack_bf16(x[8 * q + 6], x[8 * q + 7]);
            *reinterpret_cast<uint4*>(op + 8 * q) = w;
        }
    } else {
#pragma unroll
        for (int j = 0; j < 32; ++j)
            if (nb + j < N) op[j] = __float2bfloat16_rn(x[j]);
    }
}
__device__ __forceinline__ bool out_wide(const TcEpi& e) {
    return ((reinterpret_cast<uintptr_t>(e.out) & 31u) == 0) && e.ldo % 16 == 0;
}

// What a tile's epilogue needs from global memory is fetched before the tile's accumulator is
// waited for, while its mainloop runs: the biases of the warp's 128 columns into its shared
// row (HIDDEN), the ReLU mask of the thread's row as 128 bits (DX).  With biases
// and mask loaded behind the accumulator and 16-byte stores, a tile's epilogue took longer than its
// mainloop at K = 1024: the two dX launches of 16384 x 1024 outputs went from 32 + 43 us to 27 + 36,
// the HIDDEN ones from 81 + 40 to 77 + 32 (wide stores, biases and mask gave 12, 10 and 2 us of
// that pass).
__device__ __forceinline__ void hidden_bias(const TcEpi& e, int nb0, int N, float* sb) {
    const int lane = threadIdx.x & 31;
    __syncwarp();   // the previous tile's reads
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        const int n = nb0 + 32 * c + lane;
        sb[32 * c + lane] = n < N ? __ldg(e.bias + n) : 0.f;
    }
    __syncwarp();
}
__device__ __forceinline__ void dx_mask(const TcEpi& e, int row, int nb0, int M, int N, bool avec, uint32_t (&mask)[4]) {
    const __nv_bfloat16* ap = e.act + static_cast<int64_t>(row) * e.ldact + nb0;
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        mask[c] = 0;
        if (row >= M || nb0 + 32 * c >= N) continue;
        if (avec && nb0 + 32 * c + 32 <= N) {
            uint4 v[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) v[q] = *reinterpret_cast<const uint4*>(ap + 32 * c + 8 * q);
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const __nv_bfloat16* h = reinterpret_cast<const __nv_bfloat16*>(&v[q]);
#pragma unroll
                for (int t = 0; t < 8; ++t) mask[c] |= (__bfloat162float(h[t]) > 0.f ? 1u : 0u) << (8 * q + t);
            }
        } else {
            for (int j = 0; j < 32 && nb0 + 32 * c + j < N; ++j)
                mask[c] |= (__bfloat162float(ap[32 * c + j]) > 0.f ? 1u : 0u) << j;
        }
    }
}

// TC_HIDDEN: A_l = ReLU(Z_l + b_l) in bf16.
__device__ __forceinline__ void hidden_cols(const TcEpi& e, int row, int nb0, int M, int N, uint32_t taddr,
                                            const float* sb) {
    const bool wide = out_wide(e);
#pragma unroll 1
    for (int c = 0; c < 4; ++c) {
        const int nb = nb0 + 32 * c;
        if (nb >= N) break;
        uint32_t r[32];
        __syncwarp();   // lanes past M skipped the previous chunk's stores
        tc_ld_32cols(taddr + 32 * c, r);
        tc_wait_ld();
        if (row >= M) continue;
        float x[32];
#pragma unroll
        for (int j = 0; j < 32; ++j) {
            const float v = u2f(r[j]) + sb[32 * c + j];
            x[j] = v > 0.f ? v : 0.f;
        }
        store_act_chunk(e, row, nb, N, x, wide);
    }
}

// TC_DX: dZ_{l-1} = (dZ_l W_l) * 1[A_{l-1} > 0] in bf16 (a product, so a NaN stays NaN).
__device__ __forceinline__ void dx_cols(const TcEpi& e, int row, int nb0, int M, int N, uint32_t taddr,
                                        const uint32_t (&mask)[4]) {
    const bool wide = out_wide(e);
    uint32_t m0 = mask[0], m1 = mask[1], m2 = mask[2], m3 = mask[3];
#pragma unroll 1
    for (int c = 0; c < 4; ++c) {
        const int nb = nb0 + 32 * c;
        if (nb >= N) break;
        uint32_t r[32];
        __syncwarp();   // lanes past M skipped the previous chunk's stores
        tc_ld_32cols(taddr + 32 * c, r);
        tc_wait_ld();
        if (row < M) {
            float x[32];
#pragma unroll
            for (int j = 0; j < 32; ++j) x[j] = u2f(r[j]) * ((m0 >> j) & 1u ? 1.f : 0.f);
            store_act_chunk(e, row, nb, N, x, wide);
        }
        m0 = m1;
        m1 = m2;
        m2 = m3;
    }
}

// TC_GBAR: row ``row`` is an output unit; g = acc / k, w -= lr g, optional g out; returns
// the sum of g^2 over the 128 columns (fp32 per chunk, fp64 across chunks).  ``wvec``:
// w (and gbar) allow 16-byte accesses at every 32-column chunk.
__device__ __forceinline__ double gbar_cols(const TcEpi& e, int row, int nb0, int M, int N, float inv_k,
                                            uint32_t taddr, bool wvec) {
    const bool rowok = row < M;
    const int64_t at0 = e.off + static_cast<int64_t>(row) * e.ldrow + nb0;
    float* wp = e.W + at0;
    float* gp = e.gbar ? e.gbar + at0 : nullptr;
    // a chunk's 32 weights, in flight together also where the rows do not allow 16-byte loads
    // (one by one behind each other's stores they made a 1622 x 241 matrix's launch, k B = 32, 96 us; now 62)
    float4 nxt[8];
    auto fetch = [&](int c) {
        if (!rowok) return;
        if (wvec && nb0 + 32 * c + 32 <= N) {
#pragma unroll
            for (int j = 0; j < 8; ++j) nxt[j] = *reinterpret_cast<const float4*>(wp + 32 * c + 4 * j);
        } else {
            const int left = N - (nb0 + 32 * c);
            const float* p = wp + 32 * c;
#pragma unroll
            for (int j = 0; j < 8; ++j)
                nxt[j] = make_float4(4 * j < left ? p[4 * j] : 0.f, 4 * j + 1 < left ? p[4 * j + 1] : 0.f,
                                     4 * j + 2 < left ? p[4 * j + 2] : 0.f, 4 * j + 3 < left ? p[4 * j + 3] : 0.f);
        }
    };
    fetch(0);
    double sq = 0.0;
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        const int nb = nb0 + 32 * c;
        if (nb >= N) break;
        float4 cur[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) cur[j] = nxt[j];
        if (c + 1 < 4) fetch(c + 1);
        uint32_t r[32];
        __syncwarp();   // lanes past M skipped the previous chunk's stores
        tc_ld_32cols(taddr + 32 * c, r);
        tc_wait_ld();
        if (!rowok) continue;
        float part = 0.f;
        if (wvec && nb + 32 <= N) {
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                float4 g, wv = cur[q];
                g.x = u2f(r[4 * q + 0]) * inv_k;
                g.y = u2f(r[4 * q + 1]) * inv_k;
                g.z = u2f(r[4 * q + 2]) * inv_k;
                g.w = u2f(r[4 * q + 3]) * inv_k;
                wv.x = fmaf(-e.lr, g.x, wv.x);
                wv.y = fmaf(-e.lr, g.y, wv.y);
                wv.z = fmaf(-e.lr, g.z, wv.z);
                wv.w = fmaf(-e.lr, g.w, wv.w);
                *reinterpret_cast<float4*>(wp + 32 * c + 4 * q) = wv;
                if (gp) *reinterpret_cast<float4*>(gp + 32 * c + 4 * q) = g;
                part += g.x * g.x + g.y * g.y + g.z * g.z + g.w * g.w;
            }
        } else {
#pragma unroll
            for (int j = 0; j < 32; ++j) {
                if (nb + j < N) {
                    const float g = u2f(r[j]) * inv_k;
                    const float4 q = cur[j / 4];
                    const float w = j % 4 == 0 ? q.x : j % 4 == 1 ? q.y : j % 4 == 2 ? q.z : q.w;
                    wp[32 * c + j] = fmaf(-e.lr, g, w);
                    if (gp) gp[32 * c + j] = g;
                    part += g * g;
                }
            }
        }
        sq += part;
    }
    return sq;
}

// ------------------------------------------------------------------ kernel
template <int BN, int BK, int STAGES>
struct TcCfg {
    static constexpr int A_BYTES = BM * BK * 2;
    static constexpr int B_BYTES = BN * BK * 2;
    static constexpr int STAGE_BYTES = A_BYTES + B_BYTES;
    static constexpr int BAR_BYTES = 256;
    static constexpr int SMEM = STAGES * STAGE_BYTES + BAR_BYTES + 1024;   // + alignment slack
    static_assert(BK == 64 || BK == 32, "BK must be 64 or 32");
    static_assert(BN == 128 || BN == 256, "BN must be 128 or 256");
};

template <int BN, int BK, int STAGES, int KIND, int MINB>
__global__ void __launch_bounds__(kThreads, MINB)
    tc_gemm_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB, int M, int N,
                   int K, TcEpi epi, int* status) {
    grid_begin();
    static_assert(KIND == TC_DW, "the one-CTA-per-tile kernel serves the per-worker weight gradient");
    using Cfg = TcCfg<BN, BK, STAGES>;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    uint8_t* sA = smem;
    uint8_t* sB = smem + STAGES * Cfg::A_BYTES;
    uint64_t* full_bar = reinterpret_cast<uint64_t*>(smem + STAGES * Cfg::STAGE_BYTES);
    uint64_t* empty_bar = full_bar + STAGES;
    uint64_t* accum_bar = empty_bar + STAGES;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(accum_bar + 1);
    int* abort_flag = reinterpret_cast<int*>(tmem_slot + 1);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int m0 = blockIdx.y * BM, n0 = blockIdx.x * BN, z = blockIdx.z;
    const int nk = (K + BK - 1) / BK;

    if (threadIdx.x == 0) {
        for (int s = 0; s < STAGES; ++s) {
            mbar_init(smem_u32(full_bar + s), 1);
            mbar_init(smem_u32(empty_bar + s), 1);
        }
        mbar_init(smem_u32(accum_bar), 1);
        *abort_flag = 0;
        fence_mbar_init();
    }
    if (warp == 0) {
        tc_alloc(smem_u32(tmem_slot), BN);
        tc_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;

    if (warp == 0 && lane == 0) {
        // ---------------- TMA producer
        int issued = 0;
        for (int kb = 0; kb < nk; ++kb) {
            const int s = kb % STAGES;
            const uint32_t ph = (kb / STAGES) & 1;
            if (!mbar_wait(smem_u32(empty_bar + s), ph ^ 1)) {
                atomicOr(status, 1);
                atomicExch(abort_flag, 1);
                break;
            }
            if (*reinterpret_cast<volatile int*>(abort_flag)) break;
            mbar_expect_tx(smem_u32(full_bar + s), Cfg::STAGE_BYTES);
            for (int c = 0; c < BM; c += 64)
                tma_load_3d(smem_u32(sA + s * Cfg::A_BYTES + c * BK * 2), &tmA, m0 + c, kb * BK, z,
                            smem_u32(full_bar + s));
            for (int c = 0; c < BN; c += 64)
                tma_load_3d(smem_u32(sB + s * Cfg::B_BYTES + c * BK * 2), &tmB, n0 + c, kb * BK, z,
                            smem_u32(full_bar + s));
            issued = kb + 1;
        }
        if (*reinterpret_cast<volatile int*>(abort_flag)) {
            // drain this thread's copies that may still be in flight (the last STAGES issued)
            for (int kb = issued - STAGES < 0 ? 0 : issued - STAGES; kb < issued; ++kb)
                mbar_wait(smem_u32(full_bar + kb % STAGES), (kb / STAGES) & 1);
        }
    } else if (warp == 1 && lane == 0) {
        // ---------------- MMA issuer
        constexpr uint32_t idesc = instr_desc_bf16(BM, BN, true, true);
        for (int kb = 0; kb < nk; ++kb) {
            const int s = kb % STAGES;
            const uint32_t ph = (kb / STAGES) & 1;
            if (!mbar_wait(smem_u32(full_bar + s), ph)) {
                atomicOr(status, 1);
                atomicExch(abort_flag, 1);
                break;
            }
            tc_fence_after();
            const uint32_t a0 = smem_u32(sA + s * Cfg::A_BYTES);
            const uint32_t b0 = smem_u32(sB + s * Cfg::B_BYTES);
#pragma unroll
            for (int kk = 0; kk < BK / 16; ++kk) {
                if (kb * BK + 16 * kk >= K) break;   // rows past K are zero
                tc_mma(tmem, operand_desc<true, BK>(a0, kk), operand_desc<true, BK>(b0, kk), idesc,
                       (kb > 0 || kk > 0) ? 1u : 0u);
            }
            tc_commit(smem_u32(empty_bar + s));   // frees the stage once these MMAs have read it
        }
        tc_commit(smem_u32(accum_bar));           // accumulator complete (or, after an abort, quiescent)
    } else if (warp >= 2) {
        // ---------------- epilogue
        if (!mbar_wait(smem_u32(accum_bar), 0)) {
            atomicOr(status, 1);
        } else if (!*reinterpret_cast<volatile int*>(abort_flag)) {
            tc_fence_after();
            const int q = warp & 3;
            const int row = m0 + q * 32 + lane;
            const uint32_t tbase = tmem + (static_cast<uint32_t>(q * 32) << 16);
#pragma unroll 1
            for (int c = 0; c < BN / 32; ++c) {
                if (n0 + c * 32 >= N) break;
                uint32_t r[32];
                __syncwarp();
                tc_ld_32cols(tbase + c * 32, r);
                tc_wait_ld();
                epilogue_chunk<KIND>(epi, z, row, n0 + c * 32, M, N, r);
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) {
        tc_fence_after();
        tc_dealloc(tmem, BN);
    }
}

// ------------------------------------------------------------------ CTA-pair persistent kernel
// The persistent GEMM on CTA pairs: a cluster of two CTAs computes 256 x 256
// output tiles with tcgen05.mma.cta_group::2.  CTA r of the pair stages rows
// m0 + 128 r .. +127 of A and rows n0 + 128 r .. +127 of B (its half of the
// tile's B) in its own shared memory; one thread of the even CTA issues the
// MMAs, which read both CTAs' stages and accumulate output rows m0 + 128 r ..
// into CTA r's TMEM.  Per SM a 64-deep stage is 32 KB for 128 x 256 x 64 MACs,
// two thirds of what the single-CTA tile stages for the same work, so the ring
// is deeper in the same shared memory and each SM pulls fewer bytes per flop.
//
// A GBAR problem may split the K of the tiles of its last, partial round into ranges
// (choose_plan): the ranges are separate work items whose partial sums go to the workspace,
// and a later kernel of the pass adds them in range order and takes the step.  (With the
// sums in the epilogue warp that came last, a block's reads were one warp's chain of loads, and
// the code cost the other epilogues registers: the 4096-wide launches took 429 -> 525 us.  The
// launches of 4, 16 and 48 tiles at 3072-1024-1024-10, k = 96 workers of 128 samples, 192 K blocks
// a tile, went from 62 + 86 + 90 us, split only up to one round and finished by the last warp, to
// 37 + 59 + 54; the 4 rounds of 4096 x 4096 at 4096 samples, 28 tiles in the last, from 117 to 103.)
//
// One launch may carry two independent problems (nprob = 2, kinds KIND0 and KIND1).  The
// items of problem 0 are dealt to the pairs in turn; the pairs that come out one item short
// first take ``extra`` tiles of problem 1 each, and the rest of those are dealt to all.
// Shared memory: the ring of STAGES stages, 256 bytes of barriers and the order of work, then
// 128 biases per epilogue warp.
//
// Barriers (the same shared-memory offsets in both CTAs):
//   full[s]    even CTA only: its producer arrives with the byte count of both
//              CTAs' loads of stage s; the loads of both CTAs complete on it
//   empty[s]   both CTAs: the MMA issuer's commit arrives on both
//   tfull[a]   both CTAs: committed after the tile's last MMA into accumulator a
//   tempty[a]  even CTA only: the eight epilogue warps of each CTA arrive (16)
// Ten warps: 0 TMA producer and TMEM owner, 1 MMA issuer (even CTA), 2-9 epilogue:
// warp w reads TMEM lane quarter w % 4 (32 rows of the CTA's 128-row sub-tile) and
// the columns [128 h, 128 h + 128) of the tile, h = (w - 2) / 4.
constexpr int kPairThreads = 320;

struct PairProblem {
    CUtensorMap tmA, tmB;
    int M, N, K;
    TcEpi epi;
};
struct PairArgs {
    PairProblem p[2];
    int nprob;        // 1 or 2
    int max_items;    // most K ranges of problem 0 (GBAR) in all; 0: no scratch, no tile is split
    int* status;
};

// Live extent of one problem: rows past (*kdev) * kmul of the row dimension (M, or
// K for GBAR) are not computed.
struct PairShape {
    int Meff, Keff, live_k, mt_n, nt_n, msub_n, nk;
    int tiles;          // output tiles (each is 64 K elements of a matrix in memory: far below 2^31)
};
template <int KIND>
__device__ __forceinline__ PairShape pair_shape(const PairProblem& P) {
    constexpr int BN = 256, BK = 64;
    PairShape S;
    S.Meff = P.M;
    S.Keff = P.K;
    S.live_k = 1;
    if (P.epi.kdev) {
        S.live_k = *P.epi.kdev;
        const long long r = static_cast<long long>(S.live_k > 0 ? S.live_k : 0) * P.epi.kmul;
        if (KIND == TC_GBAR)
            S.Keff = r < P.K ? static_cast<int>(r) : P.K;
        else
            S.Meff = r < P.M ? static_cast<int>(r) : P.M;
    }
    S.mt_n = (S.Meff + 2 * BM - 1) / (2 * BM);
    S.nt_n = (P.N + BN - 1) / BN;
    S.msub_n = (P.M + BM - 1) / BM;   // 128-row sub-tiles of the full row extent
    S.tiles = S.live_k > 0 && S.Keff > 0 ? S.mt_n * S.nt_n : 0;
    S.nk = (S.Keff + BK - 1) / BK;
    return S;
}

// The order of the launch's work.  Items of problem 0: tiles 0 .. whole-1, then range r of tile
// whole + j as item whole + r * cut + j (cut = tiles - whole tiles of ``split`` ranges each).
struct PairPlan {
    int split, cut;         // 1, 0: no tile is split
    int whole, n0, n1;      // items of the two problems
    int hi;                 // pairs below this one have an item of problem 0 more (0: all alike)
    int extra;              // problem 1's tiles that each of the others takes first
};

// Item j of pair ``pair``: < n0 of problem 0, otherwise n0 + tile of problem 1; -1 past the end.
__device__ __forceinline__ int pair_item(const PairPlan& L, int j, int pair, int npairs) {
    const bool lo = L.hi > 0 && pair >= L.hi;
    const int c0 = L.n0 / npairs + (pair < L.hi ? 1 : 0);
    if (j < c0) return pair + j * npairs;
    j -= c0;
    const int nlo = npairs - L.hi;
    int u;
    if (lo && j < L.extra)
        u = j * nlo + pair - L.hi;
    else   // after the tiles that the pairs short of an item took first
        u = L.extra * nlo + (lo ? j - L.extra : j) * npairs + pair;
    return u < L.n1 ? L.n0 + u : -1;
}
// Tile and K range of an item of problem 0.
__device__ __forceinline__ void item_tile(const PairPlan& L, int t, int* tile, int* range) {
    *tile = t;
    *range = 0;
    if (t >= L.whole) {
        *range = (t - L.whole) / L.cut;
        *tile = L.whole + (t - L.whole) % L.cut;
    }
}
__device__ __forceinline__ int range_begin(int nk, int split, int range) {
    return split == 1 ? range * nk : static_cast<int>(static_cast<long long>(range) * nk / split);
}

// Chooses the split of the mean-gradient problem and ``extra``, one candidate (ranges s, extra)
// per lane: its K is all received samples, so with few tiles, or a nearly empty last round, a
// tile's mainloop outlasts the rest of the launch.  The estimate, in K blocks, is the later of
// a pair with an item more and one without: a split item also writes its 128 KB per CTA of
// partial sums (6), which are read back later (n / 12), and a tile
// lasts at least as long as its epilogue.
__device__ __forceinline__ PairPlan choose_plan(const PairShape& S0, const PairShape& S1, int max_items, int npairs) {
    constexpr int kEpi = 10;
    const int lane = threadIdx.x & 31;
    const int s = 1 + lane / 4, e = lane % 4;
    const int rest = S0.tiles % npairs;
    const int len = (S0.nk + s - 1) / s;
    const int item = s > 1 ? len + 6 : (len > kEpi ? len : kEpi);
    const int whole = S0.nk > kEpi ? S0.nk : kEpi, len1 = S1.nk > kEpi ? S1.nk : kEpi;
    const int n = rest * s, hi = n % npairs;
    // 0, or as many of problem 1's tiles as an item lasts (one less, one more)
    int extra = 0;
    if (e > 0 && hi > 0) {
        const int most = S1.tiles / (npairs - hi), x = item / len1 + e - 2;
        extra = x < 0 ? 0 : x < most ? x : most;
    }
    const int common = (S1.tiles - extra * (npairs - hi) + npairs - 1) / npairs;   // rounds of problem 1 over all pairs
    const long long g0 = static_cast<long long>(S0.tiles / npairs) * whole + n / npairs * item;
    const long long a = g0 + (hi > 0 ? item : 0) + static_cast<long long>(common) * len1;
    const long long b = hi > 0 ? g0 + static_cast<long long>(extra + common) * len1 : 0;
    long long cost = (a > b ? a : b) + (s > 1 ? 2 + n / 12 : 0);
    if (s > 1 && (rest == 0 || n > max_items || S0.nk < 8 * s)) cost = 1ll << 40;
    long long best = (cost << 8) | lane;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const long long x = __shfl_xor_sync(0xffffffffu, best, o);
        best = x < best ? x : best;
    }
    const int win = static_cast<int>(best & 31);
    PairPlan L;
    L.split = 1 + win / 4;
    L.extra = __shfl_sync(0xffffffffu, extra, win);
    L.hi = __shfl_sync(0xffffffffu, hi, win);
    L.cut = L.split > 1 ? rest : 0;
    L.whole = S0.tiles - L.cut;
    L.n0 = L.whole + L.cut * L.split;
    L.n1 = S1.tiles;
    return L;
}

// A split tile's partial sums: one block of 32 rows x 128 columns per (range, tile, CTA of
// the pair, epilogue warp), as float4 [chunk][quad][lane] so that a warp moves 512
// contiguous bytes per instruction.  The block of range r of split tile j is number
// (r * cut + j) * 16 + rank * 8 + warp.
constexpr int kPartFloats = kTcPartFloats;
__device__ __forceinline__ float* part_block(const TcEpi& e, const PairPlan& L, int range, int tile, int rank,
                                             int ew) {
    return e.part + (((static_cast<long long>(range) * L.cut + tile - L.whole) * 2 + rank) * 8 + ew) * kPartFloats;
}
// The first ``chunks`` 32-column chunks of this warp's TMEM block -> its partial block.
__device__ __forceinline__ void store_partial(float* dst, uint32_t taddr, int chunks, int lane) {
#pragma unroll 1
    for (int c = 0; c < chunks; ++c) {
        uint32_t r[32];
        tc_ld_32cols(taddr + 32 * c, r);
        tc_wait_ld();
#pragma unroll
        for (int q = 0; q < 8; ++q)
            reinterpret_cast<uint4*>(dst)[(c * 8 + q) * 32 + lane] =
                make_uint4(r[4 * q], r[4 * q + 1], r[4 * q + 2], r[4 * q + 3]);
    }
}

// Piece of ||g_t||^2 of one warp's block: fixed-shape warp tree, one piece per (128-row
// sub-tile, column tile, half, quarter).
__device__ __forceinline__ void store_piece(const TcEpi& e, int msub, int nt, int nt_n, bool ok, int q, int h, int lane,
                                            double sq) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) sq += __shfl_xor_sync(0xffffffffu, sq, o);
    if (lane == 0 && ok) e.pieces[(static_cast<long long>(msub) * nt_n + nt) * 8 + h * 4 + q] = sq;
}

// Fetches what the epilogue of tile t needs besides the accumulator (before it is complete).
template <int KIND>
__device__ __forceinline__ void pair_epilogue_fetch(const PairProblem& P, const PairShape& S, int t, int rank,
                                                    int q, int h, int lane, float* sb, uint32_t (&mask)[4]) {
    const int nb0 = t % S.nt_n * 256 + h * 128;
    const int row = (t / S.nt_n * 2 + rank) * BM + q * 32 + lane;
    if constexpr (KIND == TC_HIDDEN) hidden_bias(P.epi, nb0, P.N, sb);
    if constexpr (KIND == TC_DX)
        dx_mask(P.epi, row, nb0, P.M, P.N,
                ((reinterpret_cast<uintptr_t>(P.epi.act) & 15u) == 0) && P.epi.ldact % 8 == 0, mask);
}

// Epilogue of one tile for problem kind KIND (one thread: one row, 128 columns).
template <int KIND>
__device__ __forceinline__ void pair_epilogue(const PairProblem& P, const PairShape& S, int t, int rank, int q, int h,
                                              int lane, uint32_t taddr, const float* sb, const uint32_t (&mask)[4]) {
    constexpr int BN = 256;
    const TcEpi& epi = P.epi;
    const int nt = t % S.nt_n;
    const int msub = t / S.nt_n * 2 + rank;
    const int nb0 = nt * BN + h * (BN / 2);
    const int row = msub * BM + q * 32 + lane;
    if constexpr (KIND == TC_GBAR) {
        const bool wvec = ((reinterpret_cast<uintptr_t>(epi.W) & 15u) == 0) &&
                          ((reinterpret_cast<uintptr_t>(epi.gbar) & 15u) == 0) && epi.off % 4 == 0 &&
                          epi.ldrow % 4 == 0;
        double sq = gbar_cols(epi, row, nb0, P.M, P.N, 1.0f / static_cast<float>(S.live_k), taddr, wvec);
        store_piece(epi, msub, nt, S.nt_n, msub < S.msub_n, q, h, lane, sq);
    } else if constexpr (KIND == TC_DX) {
        dx_cols(epi, row, nb0, P.M, P.N, taddr, mask);
    } else if constexpr (KIND == TC_HIDDEN) {
        hidden_cols(epi, row, nb0, P.M, P.N, taddr, sb);
    } else {
#pragma unroll 1
        for (int c = 0; c < 4; ++c) {
            if (nb0 + c * 32 >= P.N) break;
            uint32_t r[32];
            __syncwarp();
            tc_ld_32cols(taddr + 32 * c, r);
            tc_wait_ld();
            epilogue_chunk<KIND>(epi, 0, row, nb0 + c * 32, P.M, P.N, r);
        }
    }
}

// One stage of this CTA's half tiles of problem kind KIND: 128 rows (or columns) of A from
// ``ma``, 128 of B from ``nb``, K block kb.
template <int KIND, int BK>
__device__ __forceinline__ void pair_load(const PairProblem& P, uint8_t* dA, uint8_t* dB, int kb, int ma, int nb,
                                          uint32_t bar) {
    if constexpr (a_mn(KIND)) {
        tma_load_2d_pair(smem_u32(dA), &P.tmA, ma, kb * BK, bar);
        tma_load_2d_pair(smem_u32(dA + BK * 128), &P.tmA, ma + 64, kb * BK, bar);
    } else {
        tma_load_2d_pair(smem_u32(dA), &P.tmA, kb * BK, ma, bar);
    }
    if constexpr (b_mn(KIND)) {
        tma_load_2d_pair(smem_u32(dB), &P.tmB, nb, kb * BK, bar);
        tma_load_2d_pair(smem_u32(dB + BK * 128), &P.tmB, nb + 64, kb * BK, bar);
    } else {
        tma_load_2d_pair(smem_u32(dB), &P.tmB, kb * BK, nb, bar);
    }
}

// The MMAs of one stage (even CTA).
template <int KIND, int BK, int BN>
__device__ __forceinline__ void pair_mma(uint32_t dcol, uint32_t a0, uint32_t b0, bool first) {
    constexpr uint32_t idesc = instr_desc_bf16(2 * BM, BN, a_mn(KIND), b_mn(KIND));
#pragma unroll
    for (int kk = 0; kk < BK / 16; ++kk)
        tc2_mma(dcol, operand_desc<a_mn(KIND), BK>(a0, kk), operand_desc<b_mn(KIND), BK>(b0, kk), idesc,
                (!first || kk > 0) ? 1u : 0u);
}

struct PairWork {
    PairShape shape[2];
    PairPlan plan;
};

template <int KIND0, int KIND1, int STAGES>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kPairThreads, 1)
    tc_gemm_pair_kernel(const __grid_constant__ PairArgs args) {
    grid_begin();
    constexpr int BN = 256, BK = 64;
    constexpr int A_BYTES = BM * BK * 2;          // 128 rows of A
    constexpr int B_BYTES = (BN / 2) * BK * 2;    // this CTA's 128 rows of B
    constexpr int STAGE_BYTES = A_BYTES + B_BYTES;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    uint8_t* sA = smem;
    uint8_t* sB = smem + STAGES * A_BYTES;
    uint64_t* full_bar = reinterpret_cast<uint64_t*>(smem + STAGES * STAGE_BYTES);
    uint64_t* empty_bar = full_bar + STAGES;
    uint64_t* tfull_bar = empty_bar + STAGES;    // [2]
    uint64_t* tempty_bar = tfull_bar + 2;        // [2]
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(tempty_bar + 2);
    int* abort_flag = reinterpret_cast<int*>(tmem_slot + 1);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t rank = cluster_rank();
    const int pair = blockIdx.x >> 1, npairs = gridDim.x >> 1;
    int* status = args.status;
    // the shapes and the order of work stay in shared memory: in registers they crowd the epilogues
    PairWork& work = *reinterpret_cast<PairWork*>(abort_flag + 1);
    static_assert((2 * STAGES + 4) * 8 + 8 + sizeof(PairWork) <= 256, "barrier block");
    if (warp == 2) {
        const PairShape a = pair_shape<KIND0>(args.p[0]);
        PairShape b{};
        if (args.nprob > 1) b = pair_shape<KIND1>(args.p[1]);
        PairPlan plan{1, 0, a.tiles, a.tiles, b.tiles, a.tiles % npairs, 0};
        if (KIND0 == TC_GBAR) plan = choose_plan(a, b, args.max_items, npairs);
        if (lane == 0) {
            if (KIND0 == TC_GBAR && blockIdx.x == 0 && args.p[0].epi.plan) {
                args.p[0].epi.plan[0] = plan.cut;
                args.p[0].epi.plan[1] = plan.split;
                args.p[0].epi.plan[2] = plan.whole;
            }
            work.shape[0] = a;
            work.shape[1] = b;
            work.plan = plan;
        }
    }
    const PairShape &S0 = work.shape[0], &S1 = work.shape[1];
    const PairPlan& L = work.plan;

    if (threadIdx.x == 0) {
        for (int s = 0; s < STAGES; ++s) {
            mbar_init(smem_u32(full_bar + s), 1);
            mbar_init(smem_u32(empty_bar + s), 1);
        }
        for (int a = 0; a < 2; ++a) {
            mbar_init(smem_u32(tfull_bar + a), 1);
            mbar_init(smem_u32(tempty_bar + a), 16);
        }
        *abort_flag = 0;
        fence_mbar_init();
    }
    if (warp == 0) {
        tc2_alloc(smem_u32(tmem_slot), 2 * BN);
        tc2_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    cluster_sync();   // both CTAs' barriers exist before any remote arrive or load completes on them
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;
    volatile int* vabort = abort_flag;

    if (warp == 0 && lane == 0) {
        // ---------------- TMA producer (both CTAs)
        long long g = 0;
        for (int j = 0, t; (t = pair_item(L, j, pair, npairs)) >= 0 && !*vabort; ++j) {
            const bool second = t >= L.n0;
            const PairShape& S = second ? S1 : S0;
            int u = t - L.n0;
            int kb0 = 0, kb1 = S.nk;
            if (!second) {
                int range;
                item_tile(L, t, &u, &range);
                if (t >= L.whole) {
                    kb0 = range_begin(S.nk, L.split, range);
                    kb1 = range_begin(S.nk, L.split, range + 1);
                }
            }
            const int ma = u / S.nt_n * (2 * BM) + static_cast<int>(rank) * BM;
            const int nb = u % S.nt_n * BN + static_cast<int>(rank) * (BN / 2);
            for (int kb = kb0; kb < kb1; ++kb, ++g) {
                const int s = static_cast<int>(g % STAGES);
                const uint32_t ph = static_cast<uint32_t>((g / STAGES) & 1);
                if (!mbar_wait(smem_u32(empty_bar + s), ph ^ 1)) {
                    atomicOr(status, 1);
                    *vabort = 1;
                    break;
                }
                if (rank == 0) mbar_expect_tx(smem_u32(full_bar + s), 2 * STAGE_BYTES);
                const uint32_t bar = map_to_rank(smem_u32(full_bar + s), 0);
                if (second)
                    pair_load<KIND1, BK>(args.p[1], sA + s * A_BYTES, sB + s * B_BYTES, kb, ma, nb, bar);
                else
                    pair_load<KIND0, BK>(args.p[0], sA + s * A_BYTES, sB + s * B_BYTES, kb, ma, nb, bar);
            }
        }
        // the last use of every stage has been consumed: no load or commit is still
        // on its way into this CTA's shared memory
        if (!*vabort) {
            for (long long q = g - STAGES < 0 ? 0 : g - STAGES; q < g; ++q) {
                if (!mbar_wait(smem_u32(empty_bar + q % STAGES), static_cast<uint32_t>((q / STAGES) & 1))) {
                    atomicOr(status, 1);
                    *vabort = 1;
                    break;
                }
            }
        }
    } else if (warp == 1 && lane == 0 && rank == 0) {
        // ---------------- MMA issuer (even CTA)
        long long g = 0;
        int i = 0;
        for (int t; (t = pair_item(L, i, pair, npairs)) >= 0 && !*vabort; ++i) {
            const bool second = t >= L.n0;
            int kb0 = 0, kb1 = second ? S1.nk : S0.nk;
            if (!second && t >= L.whole) {
                int u, range;
                item_tile(L, t, &u, &range);
                kb0 = range_begin(S0.nk, L.split, range);
                kb1 = range_begin(S0.nk, L.split, range + 1);
            }
            const int acc = i & 1;
            const uint32_t aph = static_cast<uint32_t>((i >> 1) & 1);
            if (!mbar_wait(smem_u32(tempty_bar + acc), aph ^ 1)) {
                atomicOr(status, 1);
                *vabort = 1;
                break;
            }
            tc_fence_after();
            const uint32_t dcol = tmem + static_cast<uint32_t>(acc * BN);
            bool ok = true;
            for (int kb = kb0; kb < kb1; ++kb, ++g) {
                const int s = static_cast<int>(g % STAGES);
                const uint32_t ph = static_cast<uint32_t>((g / STAGES) & 1);
                if (!mbar_wait(smem_u32(full_bar + s), ph)) {
                    atomicOr(status, 1);
                    *vabort = 1;
                    ok = false;
                    break;
                }
                tc_fence_after();
                const uint32_t a0 = smem_u32(sA + s * A_BYTES);
                const uint32_t b0 = smem_u32(sB + s * B_BYTES);
                if (second)
                    pair_mma<KIND1, BK, BN>(dcol, a0, b0, kb == kb0);
                else
                    pair_mma<KIND0, BK, BN>(dcol, a0, b0, kb == kb0);
                tc2_commit_multicast(smem_u32(empty_bar + s), 0x3);
            }
            tc2_commit_multicast(smem_u32(tfull_bar + acc), 0x3);
            if (!ok) break;
        }
    } else if (warp >= 2) {
        // ---------------- epilogue (both CTAs): 128-row sub-tile msub, lane quarter q, column half h
        const int q = warp & 3, h = (warp - 2) >> 2;
        float* sb = reinterpret_cast<float*>(smem + STAGES * STAGE_BYTES + 256) + (warp - 2) * 128;   // HIDDEN: biases
        int i = 0;
        for (int t; (t = pair_item(L, i, pair, npairs)) >= 0; ++i) {
            const int acc = i & 1;
            const uint32_t aph = static_cast<uint32_t>((i >> 1) & 1);
            uint32_t mask[4];
            if (t < L.n0)
                pair_epilogue_fetch<KIND0>(args.p[0], S0, t, static_cast<int>(rank), q, h, lane, sb, mask);
            else
                pair_epilogue_fetch<KIND1>(args.p[1], S1, t - L.n0, static_cast<int>(rank), q, h, lane, sb, mask);
            if (!mbar_wait(smem_u32(tfull_bar + acc), aph)) {
                atomicOr(status, 1);
                *vabort = 1;
                break;
            }
            if (*vabort) break;
            tc_fence_after();
            const uint32_t taddr = tmem + static_cast<uint32_t>(acc * BN + h * (BN / 2)) +
                                   (static_cast<uint32_t>(q * 32) << 16);
            if (t < L.n0) {
                if (KIND0 == TC_GBAR && t >= L.whole) {
                    int tile, range;
                    item_tile(L, t, &tile, &range);
                    const int cols = args.p[0].N - (tile % S0.nt_n * BN + h * (BN / 2));
                    const int row0 = (tile / S0.nt_n * 2 + static_cast<int>(rank)) * BM + 32 * q;
                    if (cols > 0 && row0 < args.p[0].M)
                        store_partial(part_block(args.p[0].epi, L, range, tile, static_cast<int>(rank), warp - 2),
                                      taddr, cols >= BN / 2 ? 4 : (cols + 31) / 32, lane);
                } else {
                    pair_epilogue<KIND0>(args.p[0], S0, t, static_cast<int>(rank), q, h, lane, taddr, sb, mask);
                }
            } else {
                pair_epilogue<KIND1>(args.p[1], S1, t - L.n0, static_cast<int>(rank), q, h, lane, taddr, sb, mask);
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive_remote(map_to_rank(smem_u32(tempty_bar + acc), 0));
        }
    }
    tc_fence_before();
    __syncthreads();
    if (*vabort && threadIdx.x == 0) {
        // a wait ran out: give the pair's loads and MMAs still in flight time to land
        // before the shared memory and the TMEM are released
        const uint64_t t0 = globaltimer();
        while (globaltimer() - t0 < 200000ull) {
        }
    }
    __syncthreads();
    cluster_sync();
    if (warp == 0) {
        tc_fence_after();
        tc2_dealloc(tmem, 2 * BN);
    }
}

// ------------------------------------------------------------------ persistent dW kernel
// Per-worker weight gradient G[z*ldG + m*ldrow + n] = sum_{k < K} A[z*K + k, m] B[z*K + k, n]
// (A = dZ [M, out], B = A_{l-1} [M, in], K = the worker's B samples).  The tensor maps
// are 3-D, (column, sample of the worker, worker), so that rows past a worker's K samples
// read as zero whatever K is.
//
// The kernel is bound by writing G (K is small), so it is built around that
// store.  A persistent grid (one CTA per SM) walks the tiles worker-major with n
// fastest; the MMA of tile i+1 runs into the second of two 256-column TMEM
// accumulators while the epilogue drains tile i.  Eight epilogue warps: two per
// TMEM lane quarter (32 rows of G), each owning 128 of the tile's 256 columns.
// A warp copies its 32 x 128 fp32 block TMEM -> registers -> shared memory
// (16-byte pieces XOR-swizzled by row, conflict-free) and then writes it row by
// row: each store instruction covers 512 contiguous bytes of one G row, the
// pattern that reaches the highest write bandwidth on this part.
constexpr int DW_BN = 256;
constexpr int DW_EPI_WARPS = 8;
constexpr int DW_THREADS = 32 * (2 + DW_EPI_WARPS);
constexpr int DW_WARP_COLS = 128;                         // columns of the tile per epilogue warp
constexpr int DW_STAGING_BYTES = 32 * DW_WARP_COLS * 4;   // 32 rows x 512 bytes per warp

template <int BK, int STAGES>
struct DwCfg {
    static constexpr int A_BYTES = BM * BK * 2;
    static constexpr int B_BYTES = DW_BN * BK * 2;
    static constexpr int STAGE_BYTES = A_BYTES + B_BYTES;
    static constexpr int STAGING = DW_EPI_WARPS * DW_STAGING_BYTES;
    static constexpr int BAR_BYTES = 256;
    static constexpr int SMEM = STAGES * STAGE_BYTES + STAGING + BAR_BYTES + 1024;
};

// kTest: the instantiation of the bounded-wait tests, whose MMA waits for a stage that was never
// loaded as for a lost copy.
template <int BK, int STAGES, bool kTest = false>
__global__ void __launch_bounds__(DW_THREADS, 1)
    tc_dw_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB, int Mr, int Nr,
                 int K, int batch, int* status, float* __restrict__ Gbase, int64_t ldrow, int64_t ldG, TestWaits wt) {
    grid_begin();
    const uint64_t wait_ns = kTest ? wt.limit_ns : kWaitLimitNs;
    using Cfg = DwCfg<BK, STAGES>;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    uint8_t* sA = smem;
    uint8_t* sB = smem + STAGES * Cfg::A_BYTES;
    uint8_t* staging = smem + STAGES * Cfg::STAGE_BYTES;
    uint64_t* full_bar = reinterpret_cast<uint64_t*>(staging + Cfg::STAGING);
    uint64_t* empty_bar = full_bar + STAGES;
    uint64_t* tfull_bar = empty_bar + STAGES;    // [2] accumulator ready
    uint64_t* tempty_bar = tfull_bar + 2;        // [2] accumulator drained (all epilogue warps)
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(tempty_bar + 2);
    int* abort_flag = reinterpret_cast<int*>(tmem_slot + 1);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int mt_n = (Mr + BM - 1) / BM, nt_n = (Nr + DW_BN - 1) / DW_BN;
    const int tiles_per_z = mt_n * nt_n;
    const long long total = static_cast<long long>(tiles_per_z) * batch;
    const int nk = (K + BK - 1) / BK;

    if (threadIdx.x == 0) {
        for (int s = 0; s < STAGES; ++s) {
            mbar_init(smem_u32(full_bar + s), 1);
            mbar_init(smem_u32(empty_bar + s), 1);
        }
        for (int a = 0; a < 2; ++a) {
            mbar_init(smem_u32(tfull_bar + a), 1);
            mbar_init(smem_u32(tempty_bar + a), DW_EPI_WARPS);
        }
        *abort_flag = 0;
        fence_mbar_init();
    }
    if (warp == 0) {
        tc_alloc(smem_u32(tmem_slot), 2 * DW_BN);
        tc_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;
    volatile int* vabort = abort_flag;

    if (warp == 0 && lane == 0) {
        // ---------------- TMA producer: every k block of every tile this CTA owns
        long long g = 0;
        long long issued = 0;
        for (long long t = blockIdx.x; t < total && !*vabort; t += gridDim.x) {
            const int z = static_cast<int>(t / tiles_per_z);
            const int rem = static_cast<int>(t % tiles_per_z);
            // n (out) fastest: consecutive tiles, run by neighbouring SMs at the same
            // time, fill the same G rows' line ranges together
            const int m0 = (rem / nt_n) * BM, n0 = (rem % nt_n) * DW_BN;
            for (int kb = 0; kb < nk; ++kb, ++g) {
                const int s = static_cast<int>(g % STAGES);
                const uint32_t ph = static_cast<uint32_t>((g / STAGES) & 1);
                if (!mbar_wait(smem_u32(empty_bar + s), ph ^ 1, wait_ns)) {
                    atomicOr(status, 1);
                    *vabort = 1;
                    break;
                }
                if (!(kTest && blockIdx.x == 0 && g == wt.skip_stage)) {
                    mbar_expect_tx(smem_u32(full_bar + s), Cfg::STAGE_BYTES);
#pragma unroll
                    for (int c = 0; c < BM; c += 64)
                        tma_load_3d(smem_u32(sA + s * Cfg::A_BYTES + c * BK * 2), &tmA, m0 + c, kb * BK, z,
                                    smem_u32(full_bar + s));
#pragma unroll
                    for (int c = 0; c < DW_BN; c += 64)
                        tma_load_3d(smem_u32(sB + s * Cfg::B_BYTES + c * BK * 2), &tmB, n0 + c, kb * BK, z,
                                    smem_u32(full_bar + s));
                }
                issued = g + 1;
            }
        }
        if (*vabort) {
            // the loads of the last STAGES stages may still be landing: wait for them (a
            // stage whose load never started only runs out its bound)
            for (long long q = issued - STAGES < 0 ? 0 : issued - STAGES; q < issued; ++q)
                mbar_wait(smem_u32(full_bar + q % STAGES), static_cast<uint32_t>((q / STAGES) & 1), wait_ns);
        }
    } else if (warp == 1 && lane == 0) {
        // ---------------- MMA issuer
        constexpr uint32_t idesc = instr_desc_bf16(BM, DW_BN, true, true);
        long long g = 0;
        int i = 0;
        for (long long t = blockIdx.x; t < total && !*vabort; t += gridDim.x, ++i) {
            const int acc = i & 1;
            const uint32_t aph = static_cast<uint32_t>((i >> 1) & 1);
            if (!mbar_wait(smem_u32(tempty_bar + acc), aph ^ 1, wait_ns)) {
                atomicOr(status, 1);
                *vabort = 1;
                break;
            }
            tc_fence_after();
            const uint32_t dcol = tmem + static_cast<uint32_t>(acc * DW_BN);
            bool ok = true;
            for (int kb = 0; kb < nk; ++kb, ++g) {
                const int s = static_cast<int>(g % STAGES);
                const uint32_t ph = static_cast<uint32_t>((g / STAGES) & 1);
                if (!mbar_wait(smem_u32(full_bar + s), ph, wait_ns)) {
                    atomicOr(status, 1);
                    *vabort = 1;
                    ok = false;
                    break;
                }
                tc_fence_after();
                const uint32_t a0 = smem_u32(sA + s * Cfg::A_BYTES);
                const uint32_t b0 = smem_u32(sB + s * Cfg::B_BYTES);
#pragma unroll
                for (int kk = 0; kk < BK / 16; ++kk) {
                    if (kb * BK + 16 * kk >= K) break;   // rows past K are zero
                    tc_mma(dcol, operand_desc<true, BK>(a0, kk), operand_desc<true, BK>(b0, kk), idesc,
                           (kb > 0 || kk > 0) ? 1u : 0u);
                }
                tc_commit(smem_u32(empty_bar + s));
            }
            tc_commit(smem_u32(tfull_bar + acc));
            if (!ok) break;
        }
    } else if (warp >= 2) {
        // ---------------- epilogue: TMEM -> registers -> swizzled smem -> 512-byte row stores
        const int q = warp & 3;                 // TMEM lanes 32q .. 32q+31 = G rows m0 + 32q ..
        const int half = (warp - 2) >> 2;       // columns [128 half, 128 half + 128) of the tile
        uint8_t* buf = staging + (warp - 2) * DW_STAGING_BYTES;
        int i = 0;
        for (long long t = blockIdx.x; t < total; t += gridDim.x, ++i) {
            const int acc = i & 1;
            const uint32_t aph = static_cast<uint32_t>((i >> 1) & 1);
            if (!mbar_wait(smem_u32(tfull_bar + acc), aph, wait_ns)) {
                atomicOr(status, 1);
                *vabort = 1;
                break;
            }
            if (*vabort) break;
            tc_fence_after();
            const int z = static_cast<int>(t / tiles_per_z);
            const int rem = static_cast<int>(t % tiles_per_z);
            const int m0 = (rem / nt_n) * BM, n0 = (rem % nt_n) * DW_BN;
            const uint32_t tbase = tmem + static_cast<uint32_t>(acc * DW_BN) + (static_cast<uint32_t>(q * 32) << 16);
            const int row0 = m0 + q * 32;
            const int colw = n0 + half * DW_WARP_COLS;      // first column of this warp's block
            if (row0 < Mr && colw < Nr) {
                // 1) TMEM -> smem: lane = row; 16-byte piece p of 128-byte segment sgm of row r
                //    lives at r*512 + sgm*128 + ((p ^ (r & 7)) * 16)
#pragma unroll 1
                for (int sgm = 0; sgm < DW_WARP_COLS / 32; ++sgm) {
                    uint32_t r[32];
                    tc_ld_32cols(tbase + half * DW_WARP_COLS + sgm * 32, r);
                    tc_wait_ld();
#pragma unroll
                    for (int pc = 0; pc < 8; ++pc)
                        *reinterpret_cast<uint4*>(buf + lane * 512 + sgm * 128 + ((pc ^ (lane & 7)) << 4)) =
                            make_uint4(r[4 * pc], r[4 * pc + 1], r[4 * pc + 2], r[4 * pc + 3]);
                }
                __syncwarp();
                // 2) smem -> G, one row per instruction: lane L writes columns colw + 4L .. +3
                const int sgm = lane >> 3, pc = lane & 7;
                const int col = colw + 4 * lane;
                const bool col_ok = col + 3 < Nr;   // Nr % 4 == 0 on this path: whole pieces in or out
                float* gcol = Gbase + static_cast<int64_t>(z) * ldG + col;
#pragma unroll 4
                for (int rr = 0; rr < 32; ++rr) {
                    const uint4 v = *reinterpret_cast<const uint4*>(buf + rr * 512 + sgm * 128 + ((pc ^ (rr & 7)) << 4));
                    if (col_ok && row0 + rr < Mr)
                        __stcs(reinterpret_cast<float4*>(gcol + static_cast<int64_t>(row0 + rr) * ldrow),
                               make_float4(__uint_as_float(v.x), __uint_as_float(v.y), __uint_as_float(v.z),
                                           __uint_as_float(v.w)));
                }
                __syncwarp();
            }
            // every tcgen05.ld of this accumulator has completed (wait::ld above)
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(tempty_bar + acc));
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) {
        tc_fence_after();
        tc_dealloc(tmem, 2 * DW_BN);
    }
}

// ------------------------------------------------------------------ host side
// One-shot arming of a lost load (tests of the bounded waits; see dbw_test_arm_wait_timeout).
std::atomic<long long> g_test_skip_stage{-1};
std::atomic<unsigned long long> g_test_limit_ns{0};

template <int BK, int STAGES>
cudaError_t launch_dw(const CUtensorMap& a, const CUtensorMap& b, int Mr, int Nr, int K, int batch, int* status,
                      float* gbase, int64_t ldrow, int64_t ldG, cudaStream_t st) {
    using Cfg = DwCfg<BK, STAGES>;
    const TestWaits wt = take_test_waits();
    auto kern = wt.skip_stage >= 0 ? tc_dw_kernel<BK, STAGES, true> : tc_dw_kernel<BK, STAGES, false>;
    // each CTA holds all 512 TMEM columns: ask for enough shared memory that a
    // second CTA can never be resident on the same SM (it would wait in tcgen05.alloc)
    const int smem = Cfg::SMEM > 120 * 1024 ? Cfg::SMEM : 120 * 1024;
    cudaError_t err = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (err != cudaSuccess) return err;
    const long long tiles = static_cast<long long>((Mr + BM - 1) / BM) * ((Nr + DW_BN - 1) / DW_BN) * batch;
    const int grid = static_cast<int>(tiles < sm_count() ? tiles : sm_count());
    // set up early it saves a launch gap, but its CTAs land on the SMs in the order these come
    // free and the stores of G lose their order: 256 x 4096 x 4096 (17 GB) took 6 % longer,
    // 128 x 1024 x 3072 (1.6 GB) 3 us less
    const bool early = 4.0 * batch * Mr * Nr < 4e9;
    launch_when(early, kern, grid, DW_THREADS, smem, st, a, b, Mr, Nr, K, batch, status, gbase, ldrow, ldG, wt);
    return cudaGetLastError();
}

#ifndef DBW_PAIR_STAGES
#define DBW_PAIR_STAGES 6   // TMA ring depth of the CTA-pair GEMM (32 KB per stage and CTA)
#endif

// Co-resident 2-CTA clusters of the pair kernel (the persistent grid), once per kind.
template <class Kern>
int pair_slots(Kern kern, int smem) {
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 2;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.gridDim = dim3(2 * (sm_count() / 2), 1, 1);
    cfg.blockDim = dim3(kPairThreads, 1, 1);
    cfg.dynamicSmemBytes = smem;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, kern, &cfg) != cudaSuccess || n < 1) {
        cudaGetLastError();
        n = sm_count() / 2;
    }
    return n;
}

template <int KIND0, int KIND1>
cudaError_t launch_pair(const PairArgs& args, cudaStream_t st) {
    constexpr int STAGES = DBW_PAIR_STAGES;
    constexpr int SMEM = STAGES * (2 * BM * 64 * 2) + 256 + 8 * 128 * 4 + 1024;
    static_assert(SMEM <= 227 * 1024, "pair ring does not fit in shared memory");
    auto kern = tc_gemm_pair_kernel<KIND0, KIND1, STAGES>;
    cudaError_t err = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM);
    if (err != cudaSuccess) return err;
    static int slots = 0;
    static std::once_flag once;
    std::call_once(once, [&] { slots = pair_slots(kern, SMEM); });
    long long tiles = args.max_items;   // upper bound on the items: the live extents and the plan are read on the device
    for (int i = 0; i < args.nprob; ++i)
        tiles += static_cast<long long>((args.p[i].M + 2 * BM - 1) / (2 * BM)) * ((args.p[i].N + 255) / 256);
    const int pairs = static_cast<int>(tiles < slots ? tiles : slots);
    if (pairs < 1) return cudaSuccess;
    launch(kern, 2 * pairs, kPairThreads, SMEM, st, args);
    return cudaGetLastError();
}

template <int BN, int BK, int STAGES, int KIND, int MINB>
cudaError_t launch_cfg(const CUtensorMap& a, const CUtensorMap& b, int M, int N, int K, int batch, const TcEpi& e,
                       int* status, cudaStream_t st, int min_smem) {
    using Cfg = TcCfg<BN, BK, STAGES>;
    auto kern = tc_gemm_kernel<BN, BK, STAGES, KIND, MINB>;
    const int smem = Cfg::SMEM > min_smem ? Cfg::SMEM : min_smem;
    cudaError_t err = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (err != cudaSuccess) return err;
    dim3 grid((N + BN - 1) / BN, (M + BM - 1) / BM, batch);
    launch(kern, grid, kThreads, smem, st, a, b, M, N, K, e, status);
    return cudaGetLastError();
}

}  // namespace

void arm_wait_timeout(long long stage, unsigned long long limit_ns) {
    g_test_limit_ns.store(limit_ns);
    g_test_skip_stage.store(stage);
}
TestWaits take_test_waits() {
    TestWaits wt{tcx::kWaitLimitNs, g_test_skip_stage.exchange(-1)};
    if (wt.skip_stage >= 0) wt.limit_ns = g_test_limit_ns.load();
    return wt;
}

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

static EncodeTiledFn encode_fn() {
    static EncodeTiledFn fn = nullptr;
    static std::once_flag once;
    std::call_once(once, [] {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<EncodeTiledFn>(p);
    });
    return fn;
}

// 2-D tensor map of a row-major bf16 matrix [rows, cols] with row stride ld (elements).
bool tc_make_map(CUtensorMap* tm, const void* base, int64_t rows, int64_t cols, int64_t ld, int box_rows) {
    EncodeTiledFn fn = encode_fn();
    if (!fn) return false;
    cuuint64_t dims[2] = {static_cast<cuuint64_t>(cols), static_cast<cuuint64_t>(rows)};
    cuuint64_t strides[1] = {static_cast<cuuint64_t>(ld * 2)};
    cuuint32_t box[2] = {64u, static_cast<cuuint32_t>(box_rows)};
    cuuint32_t estr[2] = {1, 1};
    return fn(tm, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides, box, estr,
              CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// The same matrix as batch blocks of rows_z rows: dimensions (column, row of the block,
// block), box 64 x box_rows x 1; rows past rows_z of a block read as zero.
static bool make_batch_map(CUtensorMap* tm, const void* base, int64_t rows_z, int64_t batch, int64_t cols, int64_t ld,
                           int box_rows) {
    EncodeTiledFn fn = encode_fn();
    if (!fn) return false;
    cuuint64_t dims[3] = {static_cast<cuuint64_t>(cols), static_cast<cuuint64_t>(rows_z),
                          static_cast<cuuint64_t>(batch)};
    cuuint64_t strides[2] = {static_cast<cuuint64_t>(ld * 2), static_cast<cuuint64_t>(rows_z * ld * 2)};
    cuuint32_t box[3] = {64u, static_cast<cuuint32_t>(box_rows), 1u};
    cuuint32_t estr[3] = {1, 1, 1};
    return fn(tm, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(base), dims, strides, box, estr,
              CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// 2-D tensor map of a row-major fp32 matrix [rows, cols] with row stride ld (elements):
// box 32 x box_rows (128-byte rows, 128-byte swizzle); reads past the extents are zero.
bool tc_make_map_f32(CUtensorMap* tm, const void* base, int64_t rows, int64_t cols, int64_t ld, int box_rows) {
    EncodeTiledFn fn = encode_fn();
    if (!fn) return false;
    cuuint64_t dims[2] = {static_cast<cuuint64_t>(cols), static_cast<cuuint64_t>(rows)};
    cuuint64_t strides[1] = {static_cast<cuuint64_t>(ld * 4)};
    cuuint32_t box[2] = {32u, static_cast<cuuint32_t>(box_rows)};
    cuuint32_t estr[2] = {1, 1};
    return fn(tm, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, const_cast<void*>(base), dims, strides, box, estr,
              CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

bool tc_make_batch_map_f32(CUtensorMap* tm, const void* base, int64_t rows, int64_t batch, int64_t cols_z, int64_t ld_z,
                           int box_rows) {
    EncodeTiledFn fn = encode_fn();
    if (!fn) return false;
    cuuint64_t dims[3] = {static_cast<cuuint64_t>(cols_z), static_cast<cuuint64_t>(batch),
                          static_cast<cuuint64_t>(rows)};
    cuuint64_t strides[2] = {static_cast<cuuint64_t>(ld_z * 4), static_cast<cuuint64_t>(batch * ld_z * 4)};
    cuuint32_t box[3] = {32u, 1u, static_cast<cuuint32_t>(box_rows)};
    cuuint32_t estr[3] = {1, 1, 1};
    return fn(tm, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 3, const_cast<void*>(base), dims, strides, box, estr,
              CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

static bool operands_ok(const TcOperands& o) {
    return encode_fn() && o.lda % 8 == 0 && o.ldb % 8 == 0 && (reinterpret_cast<uintptr_t>(o.A) & 15u) == 0 &&
           (reinterpret_cast<uintptr_t>(o.B) & 15u) == 0 && o.K >= 1;
}

// One problem of the pair kernel: 256 x 256 tiles, each CTA stages 128 rows (or columns)
// of A and 128 of B.
static int pair_problem(PairProblem* P, int kind, const TcOperands& o, const TcEpi& epi) {
    if (!operands_ok(o)) return fail(DBW_EALIGN, "tc_gemm: unsupported operand alignment");
    const bool oka = a_mn(kind) ? tc_make_map(&P->tmA, o.A, o.K, o.M, o.lda, 64)
                                : tc_make_map(&P->tmA, o.A, o.M, o.K, o.lda, BM);
    const bool okb = b_mn(kind) ? tc_make_map(&P->tmB, o.B, o.K, o.N, o.ldb, 64)
                                : tc_make_map(&P->tmB, o.B, o.N, o.K, o.ldb, 128);
    if (!oka || !okb) return fail(DBW_ECUDA, "tc_gemm: cuTensorMapEncodeTiled failed");
    P->M = o.M;
    P->N = o.N;
    P->K = o.K;
    P->epi = epi;
    return DBW_OK;
}

// A tile has at most 8 ranges, a launch at most 152: a cap on the scratch (39 MB of partial sums,
// taken per layer when the workspace is sized) that two rounds of 76 pairs reach, not a limit of the
// plan, which also holds with fewer pairs or more.
constexpr int kSplitItems = 152;
static long long gbar_tiles(int M, int N) {
    return static_cast<long long>((M + 2 * BM - 1) / (2 * BM)) * ((N + 255) / 256);
}
int tc_split_items(int M, int N) {
    const long long t = gbar_tiles(M, N) * 8;
    return static_cast<int>(t < kSplitItems ? t : kSplitItems);
}
size_t tc_split_floats(int M, int N) { return static_cast<size_t>(tc_split_items(M, N)) * 16 * kPartFloats; }

int tc_gemm_mean_dx(const TcOperands& g, const TcEpi& ge, const TcOperands& x, const TcEpi& xe, int* status,
                    cudaStream_t st) {
    PairArgs args{};
    args.nprob = 2;
    args.max_items = ge.part ? tc_split_items(g.M, g.N) : 0;
    args.status = status;
    int rc = pair_problem(&args.p[0], TC_GBAR, g, ge);
    if (rc) return rc;
    rc = pair_problem(&args.p[1], TC_DX, x, xe);
    if (rc) return rc;
    void* prof = profile_begin(PROF_GEMM, st, 0.0);
    const cudaError_t e = launch_pair<TC_GBAR, TC_DX>(args, st);
    profile_end(prof, st);
    if (e != cudaSuccess) return fail(DBW_ECUDA, "tc_gemm_mean_dx launch: %s", cudaGetErrorString(e));
    return DBW_OK;
}

int tc_dw(const TcOperands& o, int batch, const TcEpi& epi, int* status, cudaStream_t st) {
    if (!operands_ok(o)) return fail(DBW_EALIGN, "tc_dw: unsupported operand alignment");
    // 64-deep K blocks unless the worker's samples fit in one 32-deep block
    const int bk = o.K > 32 ? 64 : 32;
    CUtensorMap ta, tb;
    if (!make_batch_map(&ta, o.A, o.K, batch, o.M, o.lda, bk) || !make_batch_map(&tb, o.B, o.K, batch, o.N, o.ldb, bk))
        return fail(DBW_ECUDA, "tc_dw: cuTensorMapEncodeTiled failed");
    // algorithmic bytes: G written once (fp32), both bf16 operands read once
    const double bytes = 4.0 * batch * double(o.M) * o.N + 2.0 * batch * double(o.K) * (double(o.M) + o.N);
    float* gb = epi.G + epi.off;
    const bool vec_ok = ((reinterpret_cast<uintptr_t>(gb) & 15u) == 0) && epi.ldrow % 4 == 0 && epi.ldG % 4 == 0;
    cudaError_t e;
    void* prof = profile_begin(PROF_DW, st, bytes);
    if (!vec_ok) {
        // unaligned rows: the one-CTA-per-tile kernel (128-column tiles) with scalar stores
        e = bk == 64 ? launch_cfg<128, 64, 2, TC_DW, 4>(ta, tb, o.M, o.N, o.K, batch, epi, status, st, 48 * 1024)
                     : launch_cfg<128, 32, 2, TC_DW, 4>(ta, tb, o.M, o.N, o.K, batch, epi, status, st, 48 * 1024);
    } else {
        e = bk == 64 ? launch_dw<64, 2>(ta, tb, o.M, o.N, o.K, batch, status, gb, epi.ldrow, epi.ldG, st)
                     : launch_dw<32, 4>(ta, tb, o.M, o.N, o.K, batch, status, gb, epi.ldrow, epi.ldG, st);
    }
    profile_end(prof, st);
    if (e != cudaSuccess) return fail(DBW_ECUDA, "tc_dw launch: %s", cudaGetErrorString(e));
    return DBW_OK;
}

int tc_gemm(int kind, const TcOperands& o, const TcEpi& epi, int* status, cudaStream_t st) {
    PairArgs args{};
    args.nprob = 1;
    args.max_items = kind == TC_GBAR && epi.part ? tc_split_items(o.M, o.N) : 0;
    args.status = status;
    const int rc = pair_problem(&args.p[0], kind, o, epi);
    if (rc) return rc;
    cudaError_t e;
    void* prof = profile_begin(PROF_GEMM, st, 0.0);
    if (kind == TC_HIDDEN)
        e = launch_pair<TC_HIDDEN, TC_HIDDEN>(args, st);
    else if (kind == TC_LOGITS)
        e = launch_pair<TC_LOGITS, TC_LOGITS>(args, st);
    else if (kind == TC_GBAR)
        e = launch_pair<TC_GBAR, TC_GBAR>(args, st);
    else
        e = launch_pair<TC_DX, TC_DX>(args, st);
    profile_end(prof, st);
    if (e != cudaSuccess) return fail(DBW_ECUDA, "tc_gemm launch: %s", cudaGetErrorString(e));
    return DBW_OK;
}

}  // namespace dbw
