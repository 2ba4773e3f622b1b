"""Host-side checks of the linear algebra unit (no GPU)."""
import os
import re
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1601_02713_gb300", "csrc")


def _code(path):
    """The file without its comments."""
    with open(path) as fh:
        return re.sub(r"//[^\n]*", "", fh.read())


def test_jacobi_norm_update_is_ordered_after_every_lanes_read():
    """All lanes of a warp read a column pair's norms, lane 0 then overwrites
    them: between the two stands a warp barrier that orders memory (shuffles do
    not), outside any branch."""
    code = _code(os.path.join(CSRC, "linalg.cu"))
    read = code.index("al = nrm[p], be = nrm[q]")
    write = code.index("nrm[p] = al - tg")
    between = code[read:write]
    assert "__syncwarp();" in between
    head = between[:between.index("__syncwarp();")]
    assert head.count("{") == head.count("}") == 0


# Stands in for the CUDA runtime under the compiled unit: every launch succeeds,
# as one that is recorded into a graph does, and is printed with its cluster
# size; `room` clusters of more than 8 CTAs fit the device.
FAKE_RUNTIME = r"""
#include <cuda_runtime.h>
#include <stdio.h>
#include <stdlib.h>

namespace pimd {
struct RepMat;
void launch_jacobi(const RepMat*, int nrep, const double*, double*, double*, int ldE, double*, const int*, int,
                   cudaStream_t, int*);
}

static int room = 0;
static cudaError_t pending = cudaSuccess;
static dim3 g_grid, g_block;
static size_t g_shared;
static cudaStream_t g_stream;

static int cluster_of(const cudaLaunchConfig_t* c)
{
    for (unsigned i = 0; i < c->numAttrs; i++)
        if (c->attrs[i].id == cudaLaunchAttributeClusterDimension) return c->attrs[i].val.clusterDim.x;
    return 1;
}

extern "C" {
void** __cudaRegisterFatBinary(void*) { static void* h; return &h; }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterFunction(void**, const char*, char*, const char*, int, uint3*, uint3*, dim3*, dim3*, int*) {}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
unsigned __cudaPushCallConfiguration(dim3 g, dim3 b, size_t s, struct CUstream_st* st)
{
    g_grid = g, g_block = b, g_shared = s, g_stream = st;
    return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3* g, dim3* b, size_t* s, void* st)
{
    *g = g_grid, *b = g_block, *s = g_shared, *(cudaStream_t*)st = g_stream;
    return cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t* k, const void* f) { *k = (cudaKernel_t)f; return cudaSuccess; }
cudaError_t __cudaLaunchKernel(cudaKernel_t, dim3 g, dim3, void**, size_t, cudaStream_t)
{
    printf("%u/1 ", g.x);
    return cudaSuccess;
}
cudaError_t cudaLaunchKernel(const void*, dim3 g, dim3, void**, size_t, cudaStream_t)
{
    printf("%u/1 ", g.x);
    return cudaSuccess;
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void*, void**)
{
    printf("%u/%d ", c->gridDim.x, cluster_of(c));
    return cudaSuccess;
}
cudaError_t cudaFuncSetAttribute(const void*, enum cudaFuncAttribute, int) { return cudaSuccess; }
cudaError_t cudaOccupancyMaxActiveClusters(int* n, const void*, const cudaLaunchConfig_t* c)
{
    *n = cluster_of(c) > 8 ? room : 16;
    return cudaSuccess;
}
cudaError_t cudaGetLastError() { const cudaError_t e = pending; pending = cudaSuccess; return e; }
cudaError_t cudaPeekAtLastError() { return pending; }
cudaError_t cudaGetDevice(int* d) { *d = 0; return cudaSuccess; }
cudaError_t cudaGetSymbolAddress(void** p, const void*) { *p = nullptr; return cudaSuccess; }
}

int main(int argc, char** argv)
{
    room = atoi(argv[1]);
    pending = cudaErrorInvalidValue;   // an earlier error, which is not the solver's to clear
    for (int i = 2; i + 1 < argc; i += 2)
        pimd::launch_jacobi(nullptr, atoi(argv[i]), nullptr, nullptr, nullptr, atoi(argv[i + 1]), nullptr, nullptr, 1,
                            nullptr, nullptr);
    printf("%d\n", pending == cudaErrorInvalidValue);
    return 0;
}
"""


@pytest.fixture(scope="module")
def launches(tmp_path_factory):
    from paper_1601_02713_gb300 import build

    tmp = tmp_path_factory.mktemp("jacobi")
    build.build()
    (tmp / "fake.cpp").write_text(FAKE_RUNTIME)
    cuda = os.path.dirname(os.path.dirname(build.nvcc_path()))
    exe = str(tmp / "fake")
    subprocess.run(["g++", "-std=c++17", "-I", os.path.join(cuda, "include"), str(tmp / "fake.cpp"),
                    os.path.join(build.OBJ, "linalg.cu.o"), "-o", exe], check=True)

    def run(room, *sizes):
        out = subprocess.run([exe, str(room)] + [str(x) for s in sizes for x in s], check=True, capture_output=True,
                             text=True).stdout.split()
        assert out[-1] == "1"   # the earlier error is still pending
        return out[:-1]

    return run


@pytest.mark.parametrize("room,wide", [(8, 16), (0, 8)])
def test_jacobi_cluster_is_chosen_before_the_launch(launches, room, wide):
    """(matrices, n) -> grid / cluster size: up to 8 matrices of more than 64
    rows take 16 CTAs each where such a cluster fits and 8 where it does not,
    although no launch is refused; n of every kernel instance."""
    sizes = [(1, 65), (3, 128), (8, 192), (1, 256), (2, 384), (1, 512), (1, 768)]
    assert launches(room, *sizes) == [f"{m * wide}/{wide}" for m, _ in sizes]
    assert launches(room, (9, 65), (32, 192)) == ["72/8", "256/8"]
    assert launches(room, (1, 64), (40, 7)) == ["1/1", "40/1"]
