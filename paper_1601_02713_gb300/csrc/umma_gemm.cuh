// BF16 GEMM on the 5th-generation tensor cores (tcgen05): C[M x N] (fp32) =
// op(A) op(B), op(A)(m,k) = ta ? A[k*lda+m] : A[m*lda+k],
// op(B)(k,n) = tb ? B[n*ldb+k] : B[k*ldb+n] (bf16, row-major).
//
// One CTA of 128 threads per 128 x 128 tile of C; K in steps of 64. The
// network's products have few tiles (dW of a 256 x 256 layer: 4), so a tile is
// bound by the latency of its K steps: the operands are fetched 16 bytes at a
// time into registers while the tensor cores work on the previous step, and
// transposed there where the K direction is not the contiguous one (element by
// element into shared memory, as before, a step waited on 128 scalar loads per
// thread: a training step of 896 rows 1.06 -> 0.76 ms).
// The threads stage both operand tiles into shared memory in the canonical
// K-major, non-swizzled layout of the tensor-core descriptors (8 x 8 core
// matrices of 16-byte rows, 128 bytes each; core matrices adjacent in K are
// 128 bytes apart, those adjacent in M/N 1024 bytes apart), zero-filling past
// the edges, so any transposition and any M, N, K are handled in the copy.
// One elected thread issues four tcgen05.mma (M = 128, N = 128, K = 16 each)
// per K step into an FP32 accumulator in tensor memory and commits them to an
// mbarrier that every thread waits on (bounded) before the tiles are
// overwritten. The epilogue reads the accumulator with tcgen05.ld (warp w owns
// TMEM lanes 32w..32w+31 = rows of the tile) and stores the valid part of C.
// A wait that runs out of iterations sets *err, waits once more (bounded) for
// the MMAs in flight, frees the tensor memory and returns.
#pragma once
#include <cuda_bf16.h>
#include <stdint.h>

namespace pimd {

constexpr int UMMA_M = 128, UMMA_N = 128, UMMA_K = 64;
constexpr uint32_t UMMA_TMEM_COLS = 128;
constexpr long long UMMA_WAIT_LIMIT = 1ll << 26;

__device__ __forceinline__ uint32_t umma_smem_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

// shared-memory matrix descriptor: start address, leading (K) and stride
// (M/N) byte offsets, the fixed 0b001 field at bits 46-48, base offset 0,
// no swizzling
__device__ __forceinline__ uint64_t umma_smem_desc(uint32_t addr, uint32_t lbo, uint32_t sbo)
{
    uint64_t d = (uint64_t)((addr & 0x3FFFFu) >> 4);
    d |= (uint64_t)((lbo & 0x3FFFFu) >> 4) << 16;
    d |= (uint64_t)((sbo & 0x3FFFFu) >> 4) << 32;
    d |= (uint64_t)1 << 46;
    return d;
}

// instruction descriptor of kind::f16: FP32 accumulator (bits 4-5 = 1), A and
// B BF16 (bits 7-9, 10-12 = 1), both K-major, N >> 3 at bits 17-22, M >> 4 at
// bits 24-28
__host__ __device__ constexpr uint32_t umma_idesc_bf16(int M, int N)
{
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

__device__ __forceinline__ bool umma_wait(uint32_t bar, uint32_t phase)
{
    for (long long it = 0; it < UMMA_WAIT_LIMIT; it++) {
        uint32_t done;
        asm volatile(
            "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
            : "=r"(done)
            : "r"(bar), "r"(phase)
            : "memory");
        if (done) return true;
    }
    return false;
}

// offset (in elements) of tile element (row, k) in the core-matrix layout
__device__ __forceinline__ int umma_tile_off(int row, int k)
{
    return (((row >> 3) * (UMMA_K / 8) + (k >> 3)) << 6) + ((row & 7) << 3) + (k & 7);
}

// 8 consecutive bf16 at p, of which the first n exist (n <= 0: none); full rows
// are read in the widest pieces the address allows
__device__ __forceinline__ uint4 umma_read8(const __nv_bfloat16* p, int n)
{
    uint4 v = make_uint4(0u, 0u, 0u, 0u);
    const uintptr_t a = (uintptr_t)p;
    if (n >= 8 && (a & 15) == 0) {
        v = __ldg((const uint4*)p);
    } else if (n >= 8 && (a & 7) == 0) {
        const uint2 x = __ldg((const uint2*)p), y = __ldg((const uint2*)p + 1);
        v = make_uint4(x.x, x.y, y.x, y.y);
    } else if (n > 0) {
        unsigned w[8];
#pragma unroll
        for (int i = 0; i < 8; i++) w[i] = i < n ? (unsigned)__ldg((const unsigned short*)p + i) : 0u;
        v = make_uint4(w[0] | w[1] << 16, w[2] | w[3] << 16, w[4] | w[5] << 16, w[6] | w[7] << 16);
    }
    return v;
}

// This thread's share (64 elements) of the 128 x 64 operand tile at row r0 of R,
// k0 of K, as eight 16-byte rows of core matrices. kc: K contiguous (element
// (r, k) at P[r ld + k]), unit u = rows u & 7 of row group u >> 6, k group
// (u >> 3) & 7, eight units a thread; else (P[k ld + r]) the thread's 8 x 8 block
// of row group t & 15 and k group t >> 4, still untransposed.
__device__ __forceinline__ void umma_fetch(const __nv_bfloat16* __restrict__ P, int ld, bool kc, int r0, int R, int k0,
                                           int K, uint4 v[8])
{
    const int t = threadIdx.x;
#pragma unroll
    for (int i = 0; i < 8; i++) {
        const int u = t + 128 * i;
        const int r = r0 + (kc ? (u & 7) + 8 * (u >> 6) : 8 * (t & 15));
        const int k = k0 + (kc ? 8 * ((u >> 3) & 7) : 8 * (t >> 4) + i);
        const int left = kc ? (r < R ? K - k : 0) : (k < K ? R - r : 0);
        v[i] = left > 0 ? umma_read8(P + (kc ? (size_t)r * ld + k : (size_t)k * ld + r), left)
                        : make_uint4(0u, 0u, 0u, 0u);
    }
}

__device__ __forceinline__ void umma_put(__nv_bfloat16* s, bool kc, uint4 v[8])
{
    const int t = threadIdx.x;
    if (kc) {
#pragma unroll
        for (int i = 0; i < 8; i++) {
            const int u = t + 128 * i;
            *(uint4*)(s + umma_tile_off((u & 7) + 8 * (u >> 6), 8 * ((u >> 3) & 7))) = v[i];
        }
        return;
    }
    // transpose the 8 x 8 block: w[r] = row r, k 0..7
    uint4 w[8];
#pragma unroll
    for (int q = 0; q < 4; q++) {
        unsigned a[8], lo[4], hi[4];
#pragma unroll
        for (int k = 0; k < 8; k++) a[k] = q == 0 ? v[k].x : q == 1 ? v[k].y : q == 2 ? v[k].z : v[k].w;
#pragma unroll
        for (int m = 0; m < 4; m++) {
            lo[m] = __byte_perm(a[2 * m], a[2 * m + 1], 0x5410);
            hi[m] = __byte_perm(a[2 * m], a[2 * m + 1], 0x7632);
        }
        w[2 * q] = make_uint4(lo[0], lo[1], lo[2], lo[3]);
        w[2 * q + 1] = make_uint4(hi[0], hi[1], hi[2], hi[3]);
    }
    // every lane's block starts on the same banks: lane l stores its rows from
    // row l & 7 on (rotated in three steps, register indices constant)
#pragma unroll
    for (int b = 1; b < 8; b <<= 1) {
        const bool turn = (t & b) != 0;
        uint4 x[8];
#pragma unroll
        for (int i = 0; i < 8; i++) x[i] = turn ? w[(i + b) & 7] : w[i];
#pragma unroll
        for (int i = 0; i < 8; i++) w[i] = x[i];
    }
    const int o = umma_tile_off(8 * (t & 15), 8 * (t >> 4));
#pragma unroll
    for (int i = 0; i < 8; i++) *(uint4*)(s + o + 8 * ((i + t) & 7)) = w[i];
}

__global__ void __launch_bounds__(128) bf16_gemm_tc_kernel(int M, int N, int K, const __nv_bfloat16* __restrict__ A,
                                                           int lda, int ta, const __nv_bfloat16* __restrict__ B,
                                                           int ldb, int tb, float* __restrict__ C, int ldc, int* err)
{
    __shared__ __align__(1024) __nv_bfloat16 sA[UMMA_M * UMMA_K];
    __shared__ __align__(1024) __nv_bfloat16 sB[UMMA_N * UMMA_K];
    __shared__ __align__(8) uint64_t bar;
    __shared__ uint32_t tmem_slot;
    const int m0 = blockIdx.y * UMMA_M, n0 = blockIdx.x * UMMA_N;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t bar_a = umma_smem_addr(&bar);
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(
                         umma_smem_addr(&tmem_slot)),
                     "r"(UMMA_TMEM_COLS)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::: "memory");
    }
    if (threadIdx.x == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(bar_a) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    const uint32_t tmem = tmem_slot;
    const uint32_t idesc = umma_idesc_bf16(UMMA_M, UMMA_N);
    uint32_t phase = 0;
    bool ok = true;
    const int nk = (K + UMMA_K - 1) / UMMA_K;
    uint4 va[8], vb[8];
    umma_fetch(A, lda, !ta, m0, M, 0, K, va);
    umma_fetch(B, ldb, tb, n0, N, 0, K, vb);
    for (int kt = 0; kt < nk && ok; kt++) {
        umma_put(sA, !ta, va);
        umma_put(sB, tb, vb);
        // generic-proxy writes of the tiles -> visible to the tensor core
        asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
        __syncthreads();
        if (threadIdx.x == 0) {
            asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
#pragma unroll
            for (int kk = 0; kk < UMMA_K / 16; kk++) {
                const uint64_t ad = umma_smem_desc(umma_smem_addr(sA) + kk * 256, 128, (UMMA_K / 8) * 128);
                const uint64_t bd = umma_smem_desc(umma_smem_addr(sB) + kk * 256, 128, (UMMA_K / 8) * 128);
                const uint32_t acc = (kt > 0 || kk > 0) ? 1u : 0u;
                asm volatile(
                    "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
                    " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem),
                    "l"(ad), "l"(bd), "r"(idesc), "r"(acc)
                    : "memory");
            }
            asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(bar_a)
                         : "memory");
        }
        if (kt + 1 < nk) {
            umma_fetch(A, lda, !ta, m0, M, (kt + 1) * UMMA_K, K, va);
            umma_fetch(B, ldb, tb, n0, N, (kt + 1) * UMMA_K, K, vb);
        }
        ok = umma_wait(bar_a, phase);
        phase ^= 1u;
        // every thread saw the same barrier, so ok is uniform unless a wait
        // timed out on some threads only; make it uniform before the next copy
        ok = __syncthreads_and(ok ? 1 : 0) != 0;
    }
    if (!ok) {
        if (threadIdx.x == 0 && err) atomicExch(err, 1);
        umma_wait(bar_a, phase ^ 1u);
    } else {
        asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
        const int row = m0 + warp * 32 + lane;
        const uint32_t lane_addr = tmem + ((uint32_t)(warp * 32) << 16);
#pragma unroll 1
        for (int c0 = 0; c0 < UMMA_N; c0 += 8) {
            uint32_t v[8];
            asm volatile(
                "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];\n"
                : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7])
                : "r"(lane_addr + (uint32_t)c0));
            asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
            if (row < M)
#pragma unroll
                for (int j = 0; j < 8; j++) {
                    const int n = n0 + c0 + j;
                    if (n < N) C[(size_t)row * ldc + n] = __uint_as_float(v[j]);
                }
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    __syncthreads();
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem), "r"(UMMA_TMEM_COLS)
                     : "memory");
}

}  // namespace pimd
