// Helpers of the upsampler's tcgen05 kernels: operand layout and descriptors,
// MMA issue and completion, TMEM loads.
//
// Operand layout in shared memory: no swizzle, 8 x 8 "core matrices" of 128
// bytes (8 rows of 16 bytes); a matrix stored row by row (r, k) has its core
// matrices adjacent along k 128 bytes apart and those adjacent along r
// K/8 x 128 bytes apart (core_off).  The same bytes serve two roles:
//   K-major operand (rows are M or N, columns the reduction): leading byte
//     offset 128 (along K), stride byte offset K/8 x 128 (along M / N);
//   MN-major operand (columns are M or N, rows the reduction -- the
//     transposed matrix, without moving it): stride byte offset 128 (along
//     M / N), leading byte offset K/8 x 128 (along the reduction).
// One UMMA covers 16 elements of the reduction: two core matrices.
#pragma once
#include <cuda_bf16.h>

#include "lbt_device.cuh"
#include "lbt_mlp.h"

namespace lbt {

constexpr int kTcRows = 128;  // rows per tile (UMMA M)

__host__ __device__ constexpr int pad16(int n) { return (n + 15) / 16 * 16; }

// element (r, k) of an R x K K-major operand in the core-matrix layout
__device__ __forceinline__ int core_off(int r, int k, int K) { return (r >> 3) * (K >> 3) * 64 + (k >> 3) * 64 + (r & 7) * 8 + (k & 7); }

__device__ __forceinline__ uint32_t su32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

// shared-memory matrix descriptor: start, leading (K) and stride (M/N) byte
// offsets in 16-byte units, descriptor version 1, no swizzle
__device__ __forceinline__ uint64_t tc_desc(uint32_t addr, uint32_t lbo, uint32_t sbo)
{
    return (uint64_t)((addr >> 4) & 0x3FFF) | ((uint64_t)((lbo >> 4) & 0x3FFF) << 16) |
           ((uint64_t)((sbo >> 4) & 0x3FFF) << 32) | ((uint64_t)1 << 46);
}

// instruction descriptor of kind::f16: FP32 accumulator, bf16 A and B, A / B
// MN-major at bits 15 / 16 (else K-major), N / 8 at bit 17, M / 16 at bit 24
__device__ __forceinline__ uint32_t tc_idesc(int M, int N, bool a_mn = false, bool b_mn = false)
{
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)a_mn << 15) | ((uint32_t)b_mn << 16) |
           ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

__device__ __forceinline__ void tc_mma(uint32_t tmem_d, uint64_t da, uint64_t db, uint32_t idesc, bool acc)
{
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(tmem_d),
        "l"(da), "l"(db), "r"(idesc), "r"(acc ? 1u : 0u)
        : "memory");
}

__device__ __forceinline__ void tc_commit(uint64_t* bar)
{
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(su32(bar))
                 : "memory");
}

__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void proxy_fence() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
// 32 FP32 columns of this thread's TMEM lane, without waiting (tc_ld_wait)
__device__ __forceinline__ void tc_ld32_nowait(uint32_t taddr, uint32_t r[32])
{
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
        "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
          "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]),
          "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
          "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr));
}
__device__ __forceinline__ void tc_ld_wait() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void tc_ld16_nowait(uint32_t taddr, uint32_t r[16])
{
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
          "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr));
}

__device__ __forceinline__ void tc_ld8_nowait(uint32_t taddr, uint32_t r[8])
{
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                 : "r"(taddr));
}

// wait for a phase of the MMA barrier, giving up after about one second
__device__ __forceinline__ bool tc_wait(uint64_t* bar, uint32_t phase)
{
    uint32_t ok = 0;
    const uint64_t t0 = [] {
        uint64_t t;
        asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
        return t;
    }();
    while (true) {
        asm volatile(
            "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\tselp.u32 %0, 1, 0, p;\n\t}"
            : "=r"(ok)
            : "r"(su32(bar)), "r"(phase), "r"(20000u)
            : "memory");
        if (ok) return true;
        uint64_t t;
        asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
        if (t - t0 > 1000000000ull) return false;
    }
}

// ReLU and bf16 of two accumulators in one instruction, a in the low half
__device__ __forceinline__ uint32_t relu_bf16x2(float a, float b)
{
    uint32_t d;
    asm("cvt.rn.relu.bf16x2.f32 %0, %1, %2;" : "=r"(d) : "f"(b), "f"(a));
    return d;
}

// Columns c0 .. c0 + N - 1 of this thread's accumulator row -> ReLU, bf16 ->
// row m of a [128][128] operand.
template <int N>
__device__ __forceinline__ void relu_store(const uint32_t* r, __nv_bfloat16* h, int m, int c0)
{
#pragma unroll
    for (int g = 0; g < N; g += 8) {
        uint32_t pk[4];
#pragma unroll
        for (int j = 0; j < 4; j++) pk[j] = relu_bf16x2(__uint_as_float(r[g + 2 * j]), __uint_as_float(r[g + 2 * j + 1]));
        *reinterpret_cast<uint4*>(h + core_off(m, c0 + g, kMlpHidden)) = make_uint4(pk[0], pk[1], pk[2], pk[3]);
    }
}

// Copy a row-major [R][K] bf16 matrix into the core-matrix layout, zero rows
// from `valid` on: 16 bytes at a time (eight columns of a row are contiguous on
// both sides), element by element when the source is not 16-byte aligned.
template <int R, int K>
__device__ __forceinline__ void stage_operand(__nv_bfloat16* dst, const __nv_bfloat16* __restrict__ src, int valid, int tid,
                                              int nthr)
{
    if ((reinterpret_cast<uintptr_t>(src) & 15) == 0) {
        for (int i = tid; i < R * K / 8; i += nthr) {
            const int r = i / (K / 8), k = i % (K / 8) * 8;
            *reinterpret_cast<uint4*>(dst + core_off(r, k, K)) =
                r < valid ? __ldg(reinterpret_cast<const uint4*>(src) + i) : make_uint4(0u, 0u, 0u, 0u);
        }
    } else {
        for (int i = tid; i < R * K; i += nthr)
            dst[core_off(i / K, i % K, K)] = i / K < valid ? src[i] : __float2bfloat16(0.f);
    }
}

// A bias b as two bf16 parts hi + lo (their sum is b to 2^-16 relative).
__device__ __forceinline__ void split_bias(float b, __nv_bfloat16& hi, __nv_bfloat16& lo)
{
    hi = __float2bfloat16_rn(b);
    lo = __float2bfloat16_rn(b - __bfloat162float(hi));
}

// Biases inside the MMAs: `ones` is an A tile of ones in K columns 0 and 1,
// bias tiles are B tiles whose K columns 0 and 1 hold the parts of the bias.
__device__ __forceinline__ void stage_ones(__nv_bfloat16* ones, int tid, int nthr)
{
    for (int i = tid; i < kTcRows * 16; i += nthr)
        ones[core_off(i / 16, i % 16, 16)] = __float2bfloat16(i % 16 < 2 ? 1.f : 0.f);
}
__device__ __forceinline__ void stage_bias(__nv_bfloat16* tile, int n_pad, const float* b, int n, int tid, int nthr)
{
    for (int i = tid; i < n_pad * 16; i += nthr) {
        const int o = i / 16, k = i % 16;
        __nv_bfloat16 hi = __float2bfloat16(0.f), lo = hi;
        if (o < n && k < 2) split_bias(b[o], hi, lo);
        tile[core_off(o, k, 16)] = k == 0 ? hi : (k == 1 ? lo : __float2bfloat16(0.f));
    }
}

}  // namespace lbt
