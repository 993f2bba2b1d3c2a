// Internal helpers shared by the CUDA translation units of libdbw.
#pragma once

#include <cuda_runtime.h>
#include <cuda_bf16.h>
#include <stdint.h>

#include <utility>

#include "dbw.h"

namespace dbw {

// Records a message for dbw_last_error_string() and returns ``code``.
int fail(int code, const char* fmt, ...);
// Empties dbw_last_error_string() of the calling thread (every entry point starts with it).
void clear_error();
// Maps a pending launch error to DBW_ECUDA (with its text), else DBW_OK.
int check_launch(const char* what);
// Number of SMs of the current device (cached per device).
int sm_count();
// DBW_OK if the current device is sm_103 (compute capability 10.3), else DBW_EUNSUPPORTED.
int check_device();

// One C-ABI call: an NVTX range named after the entry point (seen by timeline tools,
// a no-op otherwise) and, with DBW_DEBUG_SYNC=1 in the environment, a
// synchronisation of the call's stream before it returns, so that an asynchronous
// fault is reported by the call that launched it (skipped while the stream is being
// captured into a graph).
class Call {
public:
    Call(const char* name, cudaStream_t st);
    ~Call();
    Call(const Call&) = delete;
    Call& operator=(const Call&) = delete;
    // rc, or DBW_ECUDA when the debug synchronisation reports an error.
    int done(int rc);

private:
    const char* name_;
    cudaStream_t st_;
};

inline bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }
inline bool aligned256(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 255u) == 0; }
inline cudaStream_t as_stream(void* s) { return reinterpret_cast<cudaStream_t>(s); }

// ----------------------------------------------------------------- kernel launches
// Every kernel of the library is launched with programmatic stream serialization: it may be
// set up while the kernel before it in the stream still runs, and its first statement,
// grid_begin(), waits until that kernel has completed and its writes are visible (a kernel
// that does not take part, such as one of the caller's, counts as a whole).  The gap between
// two dependent launches is then mostly hidden; an iteration of the small fp32 models is a
// dozen launches of 2-20 us.  A kernel that has nothing to wait for must wait all the same:
// its successor relies on it.  (us per pass without and with: 784-256-10 at n = B = 64 142 and
// 125, 784-10 at n = 16, B = 32 34.6 and 32.6, received 3072-1024-1024-10 at k = 96 501 and 477.)
// The trigger follows the wait, so that one successor at a time waits on the SMs.  With the
// trigger first, the kernels after it were set up one behind the other while the first still
// ran, and the CTAs of a small grid shared the SMs that their slots had left: an iteration of
// 400-300-200-20 at n = B = 10 in a graph took 151 us (122 now, 123 without early launches),
// 784-256-10 at n = B = 64 116 (112); 784-10 29.7 (30.2).
//
// early = false: not before its predecessor has ended.
template <class... Params, class... Args>
inline cudaError_t launch_when(bool early, void (*kern)(Params...), dim3 grid, dim3 block, size_t smem, cudaStream_t st,
                               Args&&... args) {
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = attr;
    cfg.numAttrs = early ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kern, std::forward<Args>(args)...);
}

template <class... Params, class... Args>
inline cudaError_t launch(void (*kern)(Params...), dim3 grid, dim3 block, size_t smem, cudaStream_t st,
                          Args&&... args) {
    return launch_when(true, kern, grid, block, smem, st, std::forward<Args>(args)...);
}

__device__ __forceinline__ void grid_begin() {
    cudaGridDependencySynchronize();
    cudaTriggerProgrammaticLaunchCompletion();   // the next kernel may be set up
}

// ----------------------------------------------------------------- launchers
// Selection (select.cu)
cudaError_t launch_select(const double* times, int n, const int32_t* b, int32_t* order,
                          uint8_t* mask, double* tsorted, int32_t* k_out, cudaStream_t st);

// Aggregation (aggregate.cu)
struct AggGeometry {
    int blocks;           // persistent grid size
    int rows_stride;      // n + 2: values per block in the partials
    size_t bytes;         // total partials bytes
};
AggGeometry agg_geometry(int n, int64_t d);
// flags: 0 or DBW_ALL_ROW_NORMS
cudaError_t launch_aggregate(const float* G, int64_t ld, int n, int64_t d, const uint8_t* mask,
                             float lr, float* w, float* gbar, int flags, double* partials,
                             const AggGeometry& g, cudaStream_t st);

// Estimator (estimator.cu)
cudaError_t launch_state_init(dbw_state* s, int n, int D, cudaStream_t st);
cudaError_t launch_grad_stats(const double* partials, int n, const uint8_t* mask, const float* loss,
                              const double* tsorted, double lr, dbw_state* s, double* stats_out,
                              double* row_sqnorm, cudaStream_t st);
cudaError_t launch_choose_b(dbw_state* s, double lr, double beta, int flags, int32_t* b_out,
                            double* ratio_out, const double* T_ext, cudaStream_t st);

// Push-and-wait clock and Eq. (17) (psw.cu)
size_t psw_bytes(int n);
cudaError_t launch_psw_init(void* psw, int n, cudaStream_t st);
cudaError_t launch_psw_arrivals(const void* psw, int n, const double* omega, double* e, cudaStream_t st);
cudaError_t launch_psw_record(void* psw, int n, const int32_t* order, const double* tsorted, const int32_t* k,
                              cudaStream_t st);
cudaError_t launch_psw_estimate(void* psw, int n, double tol, int max_sweeps, double* T_hat, cudaStream_t st);

// Worker gradients (grads.cu)
struct GradsPlan;
size_t grads_workspace_bytes(int L, const int32_t* widths, int n, int B, int prec);
int grads_activations(int L, const int32_t* widths, int n, int B, int prec, int layer, size_t* offset, int64_t* ld,
                      int* elem_bytes);
int launch_worker_grads(int L, const int32_t* widths, int prec, const float* w, int64_t d,
                        const float* pool, int64_t S, const int32_t* labels, const int32_t* idx,
                        int n, int B, float* G, int64_t ld, float* loss, void* ws, size_t ws_bytes,
                        cudaStream_t st);

// Tests of the bounded waits (gemm_tc.cu): the next launch of the bf16 weight gradient or of
// the wide aggregation bounds its waits by limit_ns and its first CTA does not issue the load
// of pipeline stage ``stage``; stage < 0 disarms.
void arm_wait_timeout(long long stage, unsigned long long limit_ns);
// What such a launch's kernel is given.  The production instantiations ignore it: their waits
// are bounded by tcx::kWaitLimitNs.
struct TestWaits {
    unsigned long long limit_ns;   // every mbarrier wait of the launch
    long long skip_stage;          // stage counter of block 0 left without its load; -1: none
};
// The armed test, which it disarms; skip_stage < 0 if none is.
TestWaits take_test_waits();

// Received-workers pass (grads_tc.cu)
size_t received_workspace_bytes(int L, const int32_t* widths, int n, int B, int prec);
int launch_received_grads(int L, const int32_t* widths, int prec, float* w, int64_t d, const float* pool, int64_t S,
                          const int32_t* labels, const int32_t* idx, int n, int B, const uint8_t* mask, float lr,
                          float* gbar, float* loss, double* partials, void* ws, size_t ws_bytes, cudaStream_t st);

// Partials buffer layout shared by aggregate.cu, grads_tc.cu and estimator.cu:
//   int64 header[4] = {magic, blocks, n, flags (DBW_ALL_ROW_NORMS when every row's norm is in)}
//   double sums[n + 2]              reduced totals (written by dbw_grad_stats)
//   double vals[(n + 2) * blocks]   per-block pieces, by quantity: vals[q * blocks + blk]
//                                   q < n: ||g_q||^2, q = n: SS, q = n + 1: ||g_t||^2
constexpr int64_t kPartialsMagic = DBW_PARTIALS_MAGIC;  // "DBWPART"
constexpr int kPartialsHeader = 4;
// The bits of every piece of a block of the aggregation one of whose waits ran out: a NaN that
// no arithmetic gives, so that dbw_grad_stats tells it from a NaN in the gradients.
constexpr long long kPieceTimedOut = 0x7ff8444257544f21ll;

}  // namespace dbw
