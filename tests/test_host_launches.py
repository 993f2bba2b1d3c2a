"""What the host code launches, checked without a GPU: the library's objects are linked
against a stand-in for the CUDA runtime.

The opt-in to more than 48 KB of shared memory belongs to the kernel, not to a launch, and
host threads share it: a call that sets it to its own need would let a second thread, whose
n is smaller, lower it between this thread's set and its launch, which the runtime then
refuses.  The stand-in keeps the opt-in of each kernel, refuses a launch above it as the
runtime does, and before each launch makes the call of the second thread.

The selection runs in several CTAs that share nothing; where an output lies over an input
that each of them reads, it takes one."""
import ctypes as C
import os
import subprocess

import pytest

from paper_2004_14696_gb300 import build as B
from paper_2004_14696_gb300 import dbw

RUNTIME = r"""
#include <cuda_runtime_api.h>
enum { kMost = 256, kDefault = 48 * 1024 };
static const void* func[kMost];
static int limit[kMost], used, inside;
static cudaError_t last;
int launches, refused, grid;
void (*other_thread)(void);

static int* limit_of(const void* f) {
    int i = 0;
    while (i < used && func[i] != f) ++i;
    if (i == used) { func[used] = f; limit[used++] = kDefault; }
    return &limit[i];
}
cudaError_t cudaFuncSetAttribute(const void* f, enum cudaFuncAttribute attr, int value) {
    if (attr == cudaFuncAttributeMaxDynamicSharedMemorySize) *limit_of(f) = value;
    return cudaSuccess;
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void* f, void** args) {
    if (other_thread && !inside) {
        inside = 1;
        other_thread();
        inside = 0;
    }
    ++launches;
    grid = c->gridDim.x;
    if (c->dynamicSmemBytes > (size_t)*limit_of(f)) {
        ++refused;
        return last = cudaErrorInvalidValue;
    }
    return cudaSuccess;
}
cudaError_t cudaGetLastError(void) { cudaError_t e = last; last = cudaSuccess; return e; }
const char* cudaGetErrorString(cudaError_t e) { return e ? "refused" : "no error"; }
cudaError_t cudaGetDevice(int* d) { *d = 0; return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, enum cudaDeviceAttr a, int d) {
    *v = a == cudaDevAttrComputeCapabilityMajor ? 10 : a == cudaDevAttrComputeCapabilityMinor ? 3 : 152;
    return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* n, const void* f, int t, size_t s, unsigned g) {
    *n = 2;
    return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveClusters(int* n, const void* f, const cudaLaunchConfig_t* c) { *n = 76; return cudaSuccess; }
cudaError_t cudaMemsetAsync(void* p, int v, size_t n, cudaStream_t s) { return cudaSuccess; }
cudaError_t cudaGetSymbolAddress(void** p, const void* s) { *p = (void*)s; return cudaSuccess; }
cudaError_t cudaGetDriverEntryPointByVersion(const char* s, void** p, unsigned v, unsigned long long f,
                                             enum cudaDriverEntryPointQueryResult* r) { return cudaErrorUnknown; }
cudaError_t cudaEventCreate(cudaEvent_t* e) { return cudaErrorUnknown; }
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t s) { return cudaErrorUnknown; }
cudaError_t cudaEventSynchronize(cudaEvent_t e) { return cudaErrorUnknown; }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t a, cudaEvent_t b) { return cudaErrorUnknown; }
cudaError_t cudaStreamIsCapturing(cudaStream_t s, enum cudaStreamCaptureStatus* c) { return cudaErrorUnknown; }
cudaError_t cudaStreamSynchronize(cudaStream_t s) { return cudaErrorUnknown; }
/* what the compiler's registration code calls */
static void* handle;
void** __cudaRegisterFatBinary(void* fat) { return &handle; }
void __cudaRegisterFatBinaryEnd(void** h) {}
void __cudaUnregisterFatBinary(void** h) {}
void __cudaRegisterFunction(void** h, const char* f, char* df, const char* dn, int t, void* a, void* b, void* c, void* d,
                            int* w) {}
void __cudaRegisterVar(void** h, char* v, char* da, const char* dn, int e, size_t s, int c, int g) {}
unsigned __cudaPopCallConfiguration(void* g, void* b, size_t* s, void* st) { return 0; }
cudaError_t __cudaGetKernel(void* k, const void* f) { return cudaErrorUnknown; }
cudaError_t __cudaLaunchKernel(void* k, ...) { return cudaErrorUnknown; }
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    B.build()
    objs = [os.path.join(B.BUILD, s[:-3] + ".o") for s in B.sources()]
    if not all(os.path.exists(o) for o in objs):
        B.build(force=True)
    tmp = tmp_path_factory.mktemp("runtime")
    src, out = tmp / "runtime.c", tmp / "libdbw_on_stand_in.so"
    src.write_text(RUNTIME)
    cuda = os.path.join(os.path.dirname(os.path.dirname(B.nvcc())), "include")
    subprocess.run(["gcc", "-w", "-fPIC", "-I", cuda, "-c", str(src), "-o", str(tmp / "runtime.o")], check=True)
    subprocess.run(["g++", "-shared", "-Wl,-Bsymbolic", "-o", str(out), str(tmp / "runtime.o"), *objs, "-ldl"], check=True)
    L = C.CDLL(str(out))
    for name, (res, args) in dbw._SIGS.items():
        getattr(L, name).restype, getattr(L, name).argtypes = res, args
    return L


def with_other_thread(lib, call, other):
    hook = C.CFUNCTYPE(None)(other)
    C.c_void_p.in_dll(lib, "other_thread").value = C.cast(hook, C.c_void_p).value
    launches, refused = C.c_int.in_dll(lib, "launches"), C.c_int.in_dll(lib, "refused")
    launches.value = refused.value = 0
    try:
        rc = call()
    finally:
        C.c_void_p.in_dll(lib, "other_thread").value = None
    assert launches.value > 0
    assert not refused.value, lib.dbw_last_error_string()
    return rc


@pytest.mark.parametrize("flags", [0, dbw.ALL_ROW_NORMS])
@pytest.mark.parametrize("d", [100_000, 10_000_000])
@pytest.mark.parametrize("n,other", [(256, 16), (1024, 256), (16, 1024)])
def test_two_threads_aggregate(lib, n, other, d, flags):
    # the second thread only asks for its buffer's size, or aggregates as well
    part = lib.dbw_aggregate_partials_bytes(n, d)

    def aggregate(n, bytes_):
        return lib.dbw_aggregate_update(256, d, n, d, 256, C.c_float(0.1), 256, None, flags, 256, bytes_, None)
    for second in (lambda: lib.dbw_aggregate_partials_bytes(other, d),
                   lambda: aggregate(other, lib.dbw_aggregate_partials_bytes(other, d))):
        assert with_other_thread(lib, lambda: aggregate(n, part), second) == dbw.DBW_OK


@pytest.mark.parametrize("n,other", [(256, 16), (1024, 40), (40, 1024)])
def test_two_threads_fit(lib, n, other):
    def fit(n):
        return lib.dbw_psw_estimate(256, n, C.c_double(1e-4), 10, 256, None)
    assert with_other_thread(lib, lambda: fit(n), lambda: fit(other)) == dbw.DBW_OK


@pytest.mark.parametrize("n", [1, 8, 9, 256, 1024])
def test_selection_over_its_own_inputs_is_one_cta(lib, n):
    times, b, order, mask, out, k = 1 << 20, 2 << 20, 3 << 20, 4 << 20, 5 << 20, 6 << 20   # addresses, not read here
    grid = C.c_int.in_dll(lib, "grid")

    def ctas(times, b, tsorted, k_out):
        grid.value = 0
        assert lib.dbw_select_fastest(times, n, b, order, mask, tsorted, k_out, None) == dbw.DBW_OK
        return grid.value
    assert ctas(times, b, out, k) == ctas(times, b, out, None) == -(-n // 8)
    assert ctas(times, b, times, k) == 1          # sorted in place
    assert ctas(times, b, times + 8 * n - 8, k) == 1 and ctas(times + 8 * n - 8, b, times, k) == 1
    assert ctas(times, b, out, b) == 1            # k over b: a CTA could read b after another's k
