"""Device memory of the float-float copies, without a GPU: the library linked to
a stand-in runtime whose kernels do nothing and whose device holds a given number
of bytes. The copies take only what the rest of a call leaves."""
import os
import subprocess

import pytest

MAIN = r"""
#include <cuda_runtime.h>
#include <stdio.h>
#include <stdlib.h>
#include <string.h>

#include <map>
#include <vector>

#include "pimdgb.h"

static std::map<void*, size_t> held;
static size_t used = 0, peak = 0, room = (size_t)1 << 40;

extern "C" {
cudaError_t cudaMalloc(void** p, size_t n)
{
    if (used + n > room) return cudaErrorMemoryAllocation;
    *p = calloc(n, 1);
    held[*p] = n;
    used += n;
    if (used > peak) peak = used;
    return cudaSuccess;
}
cudaError_t cudaFree(void* p)
{
    if (!p) return cudaSuccess;
    if (!held.count(p)) abort();
    used -= held[p];
    held.erase(p);
    free(p);
    return cudaSuccess;
}
static cudaError_t copy(void* d, const void* s, size_t n) { memcpy(d, s, n); return cudaSuccess; }
cudaError_t cudaMemcpy(void* d, const void* s, size_t n, cudaMemcpyKind) { return copy(d, s, n); }
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind, cudaStream_t) { return copy(d, s, n); }
cudaError_t cudaMemset(void* d, int v, size_t n) { memset(d, v, n); return cudaSuccess; }
cudaError_t cudaMemsetAsync(void* d, int v, size_t n, cudaStream_t) { memset(d, v, n); return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr, int) { *v = 152; return cudaSuccess; }
cudaError_t cudaGetDevice(int* d) { *d = 0; return cudaSuccess; }
cudaError_t cudaGetDeviceCount(int* n) { *n = 1; return cudaSuccess; }
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaDeviceSynchronize() { return cudaSuccess; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
cudaError_t cudaPeekAtLastError() { return cudaSuccess; }
const char* cudaGetErrorString(cudaError_t) { return "error"; }
cudaError_t cudaEventCreate(cudaEvent_t*) { return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t*, unsigned) { return cudaSuccess; }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) { *ms = 0; return cudaSuccess; }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t*, unsigned) { return cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) { return cudaErrorNotSupported; }
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t*) { return cudaErrorNotSupported; }
cudaError_t cudaGraphInstantiate(cudaGraphExec_t*, cudaGraph_t, unsigned long long) { return cudaErrorNotSupported; }
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) { return cudaErrorNotSupported; }
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }
cudaError_t cudaFuncSetAttribute(const void*, enum cudaFuncAttribute, int) { return cudaSuccess; }
cudaError_t cudaOccupancyMaxActiveClusters(int* n, const void*, const cudaLaunchConfig_t*) { *n = 8; return cudaSuccess; }
cudaError_t cudaGetSymbolAddress(void** p, const void*) { *p = nullptr; return cudaSuccess; }
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t*, const void*, void**) { return cudaSuccess; }
cudaError_t cudaLaunchKernel(const void*, dim3, dim3, void**, size_t, cudaStream_t) { return cudaSuccess; }
cudaError_t __cudaLaunchKernel(cudaKernel_t, dim3, dim3, void**, size_t, cudaStream_t) { return cudaSuccess; }
cudaError_t __cudaGetKernel(cudaKernel_t* k, const void* f) { *k = (cudaKernel_t)f; return cudaSuccess; }
void** __cudaRegisterFatBinary(void*) { static void* h; return &h; }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterFunction(void**, const char*, char*, const char*, int, uint3*, uint3*, dim3*, dim3*, int*) {}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
unsigned __cudaPushCallConfiguration(dim3, dim3, size_t, struct CUstream_st*) { return 0; }
cudaError_t __cudaPopCallConfiguration(dim3* g, dim3* b, size_t* s, void* st)
{
    *g = *b = dim3(1), *s = 0, *(cudaStream_t*)st = 0;
    return cudaSuccess;
}
}

// Fock builds of n[0], n[1], ... replicas of one p atom on one context; the peak
// above what the context holds, or 0 for a failed call
static size_t calls(double tight, const std::vector<int>& n, size_t limit)
{
    // tight: the exponent of an element that no molecule holds (1e9: FP64 only)
    const int Z[2] = {2, 4}, nsh[2] = {3, 1}, l[4] = {0, 1, 1, 0}, np[4] = {1, 1, 1, 1};
    const double ex[4] = {1.0, 0.5, 1.5, tight}, co[4] = {1, 1, 1, 1};
    pimd_ctx* ctx;
    pimd_basis* bas;
    room = (size_t)1 << 40;
    if (pimd_ctx_create(&ctx, 0) || pimd_basis_create(&bas, 2, Z, nsh, l, np, ex, co, 1)) abort();
    const size_t base = used;
    peak = used;
    if (limit) room = base + limit;
    bool ok = true;
    for (int k : n) {
        std::vector<double> X(3 * k, 0.0), D(49 * k), G(49 * k);
        const int z = 2;
        ok = ok && pimd_fock_dev(ctx, k, 1, &z, X.data(), bas, 1e-12, 0.0, D.data(), G.data()) == PIMD_OK;
    }
    const size_t p = peak - base;
    pimd_basis_destroy(bas);
    pimd_ctx_destroy(ctx);
    return ok ? p : 0;
}

int main()
{
    for (const std::vector<int>& n : {std::vector<int>{4000}, std::vector<int>{1000, 4000}}) {
        const size_t fp64 = calls(1e9, n, 0), all = calls(1.0, n, 0);
        printf("%zu %zu %zu %zu %zu\n", fp64, all, calls(1.0, n, fp64), calls(1.0, n, (fp64 + all) / 2),
               calls(1.0, n, fp64 - 1));
    }
    return 0;
}
"""


@pytest.fixture(scope="module")
def rows(tmp_path_factory):
    from paper_1601_02713_gb300 import build

    tmp = tmp_path_factory.mktemp("memory")
    build.build()
    (tmp / "main.cpp").write_text(MAIN)
    cuda = os.path.dirname(os.path.dirname(build.nvcc_path()))
    exe = str(tmp / "main")
    units = build.HAND_WRITTEN + [os.path.basename(u) for u in build.generate_sources()]
    objs = [os.path.join(build.OBJ, u + ".o") for u in units]
    subprocess.run(["g++", "-std=c++17", "-w", "-I", os.path.join(cuda, "include"), "-I", build.INCLUDE,
                    str(tmp / "main.cpp")] + objs + ["-o", exe], check=True)
    out = subprocess.run([exe], check=True, capture_output=True, text=True, timeout=300).stdout
    return [[int(x) for x in row.split()] for row in out.splitlines()]


@pytest.mark.parametrize("k", [0, 1])
def test_a_call_that_fits_in_fp64_is_not_refused(rows, k):
    """One call, and one after a smaller one whose copies are still held."""
    fp64, all_, tight, between, less = rows[k]
    assert all_ > 1.1 * fp64   # the copies are made where there is room
    assert 0 < tight <= fp64
    assert 0 < between < all_
    assert less == 0           # the stand-in's limit holds


def test_calls_in_fp64_make_no_copies(rows):
    """The pair data of a call that stays in FP64: 12 fields in FP64 and FP32 of
    up to nine primitive pairs, per shell pair (6 of the atom's 3 shells)."""
    fp64, all_ = rows[0][:2]
    per_pair = (all_ - fp64) / (4000 * 6)
    copies = 15 * 9 * 8 + 3 * 8 + 8 * 49 / 6   # ppd, abd and the density
    assert abs(per_pair - copies) < 0.01 * copies
