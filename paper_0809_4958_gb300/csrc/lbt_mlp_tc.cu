// Forward of the learned boundary upsampler on the fifth-generation tensor
// cores (tcgen05): 128-row tiles, the three layers as UMMA instructions with
// bf16 operands in shared memory and FP32 accumulators in tensor memory
// (TMEM), bias + ReLU + bf16 epilogues read back with tcgen05.ld.  Operand
// layout and helpers: lbt_tc.cuh; training: lbt_mlp_train.cu.
#include <cstdio>

#include "lbt_tc.cuh"

namespace lbt {

namespace {

// Forward: four groups of four warps per block (one block per SM), each
// group with its own 128-row tile, activations in shared memory, 128 TMEM
// columns and MMA barrier, so that four tiles are in flight per SM and a
// group's epilogue overlaps the other groups' MMAs.
constexpr int kFwGroups = 4;
constexpr int kFwThreads = kFwGroups * kTcRows;
constexpr int kFwCols = kFwGroups * kMlpHidden;  // 512: the whole TMEM of the SM

template <int NOUT>
struct TcSmem {
    static constexpr int kNP = pad16(NOUT);
    __nv_bfloat16 w1[kMlpHidden * kMlpIn];
    __nv_bfloat16 w2[kMlpHidden * kMlpHidden];
    __nv_bfloat16 w3[kNP * kMlpHidden];
    __nv_bfloat16 x[kFwGroups][kTcRows * kMlpIn];
    __nv_bfloat16 h[kFwGroups][kTcRows * kMlpHidden];
    // biases inside the MMAs: an A tile of ones in K columns 0 and 1, and B
    // tiles whose K columns 0 and 1 hold the FP32 bias split into bf16
    // high and low parts (their sum is the bias to 2^-16 relative); layer 1
    // uses feature columns 24 and 25 (zero padding) and rows 24, 25 of W1
    __nv_bfloat16 ones[kTcRows * 16];
    __nv_bfloat16 bb2[kMlpHidden * 16];
    __nv_bfloat16 bb3[kNP * 16];
    uint64_t bar[kFwGroups];
    uint32_t tmem;
};
static_assert(sizeof(TcSmem<48>) <= 227 * 1024, "forward shared memory");

// barrier over the 128 threads of one forward group (ids 1 .. 4; 0 is __syncthreads)
__device__ __forceinline__ void group_sync(int g) { asm volatile("bar.sync %0, %1;" ::"r"(g + 1), "r"(kTcRows) : "memory"); }
__device__ __forceinline__ bool group_all(int g, bool v)
{
    uint32_t r;
    asm volatile(
        "{\n\t.reg .pred pi, po;\n\tsetp.ne.u32 pi, %1, 0;\n\tbarrier.cta.red.and.pred po, %2, %3, pi;\n\t"
        "selp.u32 %0, 1, 0, po;\n\t}"
        : "=r"(r)
        : "r"((uint32_t)v), "r"(g + 1), "r"(kTcRows)
        : "memory");
    return r != 0;
}

// accumulator columns [0, 128) of this thread's row (the bias is already in
// them) -> ReLU, bf16 -> row m of the next layer's A operand
// (64 columns per round: two 32-column TMEM loads in flight, one wait)
__device__ __forceinline__ void hidden_epilogue(uint32_t tmem_row, __nv_bfloat16* h, int m)
{
#pragma unroll 1
    for (int c0 = 0; c0 < kMlpHidden; c0 += 64) {
        uint32_t r[64];
        tc_ld32_nowait(tmem_row + c0, r);
        tc_ld32_nowait(tmem_row + c0 + 32, r + 32);
        tc_ld_wait();
        relu_store<64>(r, h, m, c0);
    }
}

template <int NOUT>
__global__ void __launch_bounds__(kFwThreads, 1) k_mlp_forward_tc(const __nv_bfloat16* __restrict__ X, int64_t rows,
                                                                  const unsigned char* __restrict__ params, MlpLayout L,
                                                                  float* __restrict__ Y, int64_t col_stride,
                                                                  int32_t* err)
{
    using Sm = TcSmem<NOUT>;
    constexpr int NP = Sm::kNP;
    extern __shared__ __align__(128) unsigned char tc_smem_raw[];
    Sm& sm = *reinterpret_cast<Sm*>(tc_smem_raw);
    const int tid = threadIdx.x, warp = tid >> 5;
    const int g = warp / 4;          // group: its tile, buffers, TMEM columns and barrier
    const int q = warp % 4;          // TMEM lane quadrant this warp reads
    const int m = 32 * q + (tid & 31);  // row of the group's tile this thread owns
    const int gt = tid % kTcRows;    // thread index within the group

    // weights into the core-matrix layout (W3 padded with zero rows to NP), once per block
    stage_operand<kMlpHidden, kMlpIn>(sm.w1, reinterpret_cast<const __nv_bfloat16*>(params + L.w1), kMlpHidden, tid, kFwThreads);
    stage_operand<kMlpHidden, kMlpHidden>(sm.w2, reinterpret_cast<const __nv_bfloat16*>(params + L.w2), kMlpHidden, tid,
                                          kFwThreads);
    stage_operand<NP, kMlpHidden>(sm.w3, reinterpret_cast<const __nv_bfloat16*>(params + L.w3), NOUT, tid, kFwThreads);
    __syncthreads();  // W1 rows 24, 25 are overwritten below
    const float* b1 = reinterpret_cast<const float*>(params + L.b1);
    for (int n = tid; n < kMlpHidden; n += kFwThreads)  // layer 1: feature columns 24, 25 are set to one at staging
        split_bias(b1[n], sm.w1[core_off(n, kMlpFeat, kMlpIn)], sm.w1[core_off(n, kMlpFeat + 1, kMlpIn)]);
    stage_ones(sm.ones, tid, kFwThreads);
    stage_bias(sm.bb2, kMlpHidden, reinterpret_cast<const float*>(params + L.b2), kMlpHidden, tid, kFwThreads);
    stage_bias(sm.bb3, NP, reinterpret_cast<const float*>(params + L.b3), NOUT, tid, kFwThreads);
    if (tid < kFwGroups) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(su32(&sm.bar[tid])) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(su32(&sm.tmem)),
                     "r"(kFwCols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    proxy_fence();
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    // the group's 128 columns hold the hidden accumulators of layers 1 and 2
    // and then the output (each written after the previous epilogue read it)
    const uint32_t tmem_g = sm.tmem + (uint32_t)(kMlpHidden * g);
    const uint32_t tmem_row = tmem_g + ((uint32_t)(32 * q) << 16);
    const uint32_t id_h = tc_idesc(kTcRows, kMlpHidden), id_o = tc_idesc(kTcRows, NP);
    const uint32_t ax = su32(sm.x[g]), ah = su32(sm.h[g]), a1 = su32(sm.w1), a2 = su32(sm.w2), a3 = su32(sm.w3);
    const uint32_t a_one = su32(sm.ones), ab2 = su32(sm.bb2), ab3 = su32(sm.bb3);
    constexpr uint32_t kLbo = 128, kSbo16 = (16 / 8) * 128, kSbo32 = (kMlpIn / 8) * 128,
                       kSbo128 = (kMlpHidden / 8) * 128;
    uint32_t phase = 0;
    bool ok = true;

    const int64_t ntiles = (rows + kTcRows - 1) / kTcRows;
    const int64_t stride = (int64_t)gridDim.x * kFwGroups;
    // features of a tile, row m = this thread (zeros past the last row); the
    // next tile's are loaded into registers while this one is computed
    uint4 xr[kMlpIn / 8];
    auto load_x = [&](int64_t tile) {
        const int64_t r = tile * kTcRows + m;
        const bool in = tile < ntiles && r < rows;
        const uint4* src = reinterpret_cast<const uint4*>(X + (in ? r : 0) * kMlpIn);
#pragma unroll
        for (int c = 0; c < kMlpIn / 8; c++) xr[c] = in ? __ldg(src + c) : make_uint4(0u, 0u, 0u, 0u);
        // feature columns 24 and 25 (zero padding) carry the ones of layer 1's bias
        static_assert(kMlpFeat == 24, "the bias columns follow the 24 features");
        xr[3].x = 0x3F803F80u;  // bf16 1.0 in both halves
    };
    int64_t tile = (int64_t)blockIdx.x * kFwGroups + g;
    load_x(tile);
    for (; tile < ntiles && ok; tile += stride) {
        const int64_t r0 = tile * kTcRows;
#pragma unroll
        for (int c = 0; c < kMlpIn / 8; c++) *reinterpret_cast<uint4*>(sm.x[g] + core_off(m, 8 * c, kMlpIn)) = xr[c];
        load_x(tile + stride);
        // the three layers; each: MMAs by one thread of the group, commit, wait, epilogue
        for (int layer = 0; layer < 3 && ok; layer++) {
            proxy_fence();  // generic-proxy shared-memory writes -> tensor-core reads
            tc_fence_before();
            group_sync(g);
            tc_fence_after();
            if (gt == 0) {
                if (layer == 0) {
                    for (int ks = 0; ks < kMlpIn / 16; ks++)
                        tc_mma(tmem_g, tc_desc(ax + ks * 256, kLbo, kSbo32), tc_desc(a1 + ks * 256, kLbo, kSbo32), id_h,
                               ks > 0);
                } else {
                    const uint32_t ab = layer == 1 ? a2 : a3;
                    const uint32_t id = layer == 1 ? id_h : id_o;
                    for (int ks = 0; ks < kMlpHidden / 16; ks++)
                        tc_mma(tmem_g, tc_desc(ah + ks * 256, kLbo, kSbo128), tc_desc(ab + ks * 256, kLbo, kSbo128), id,
                               ks > 0);
                    // + ones x (bias hi, lo): the layer's bias
                    tc_mma(tmem_g, tc_desc(a_one, kLbo, kSbo16), tc_desc(layer == 1 ? ab2 : ab3, kLbo, kSbo16), id, true);
                }
                tc_commit(&sm.bar[g]);
            }
            const bool arrived = tc_wait(&sm.bar[g], phase);
            phase ^= 1u;
            if (!group_all(g, arrived)) {
                ok = false;  // the MMAs did not complete within a second
                break;
            }
            tc_fence_after();
            if (layer < 2) {
                hidden_epilogue(tmem_row, sm.h[g], m);
            } else {
                // every lane takes part in the (warp-collective) TMEM loads;
                // rows past the end store nothing
                const bool in = r0 + m < rows;
                static_assert(NP == 32 || NP == 48, "output columns: one 32-column load and at most one 16-column one");
                uint32_t r[NP];  // every output column in flight at once, one wait
                tc_ld32_nowait(tmem_row, r);
                if constexpr (NP == 48) tc_ld16_nowait(tmem_row + 32, r + 32);
                tc_ld_wait();
#pragma unroll
                for (int c0 = 0; c0 < NP; c0 += 16) {
                    float v[16];
#pragma unroll
                    for (int j = 0; j < 16; j++) v[j] = __uint_as_float(r[c0 + j]);
                    if (col_stride == 0) {  // row-major [rows][NOUT]: four 16-byte stores per lane
                        float* y = Y + (r0 + m) * NOUT;
#pragma unroll
                        for (int j = 0; j < 16; j += 4)
                            if (in && c0 + j < NOUT)
                                *reinterpret_cast<float4*>(y + c0 + j) = make_float4(v[j], v[j + 1], v[j + 2], v[j + 3]);
                    } else {  // column-major Y[col * col_stride + row]: the warp's 32 rows in one line per column
#pragma unroll
                        for (int j = 0; j < 16; j++)
                            if (in && c0 + j < NOUT) Y[(int64_t)(c0 + j) * col_stride + r0 + m] = v[j];
                    }
                }
            }
        }
    }
    if (!ok) {
        if (gt == 0 && err) atomicCAS(err, 0, LB_ERR_TIMEOUT);
        tc_wait(&sm.bar[g], phase ^ 1u);  // let an MMA still in flight finish (bounded)
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(sm.tmem), "r"(kFwCols) : "memory");
}

template <int NOUT>
cudaError_t forward_tc(const void* X, int64_t rows, const void* params, const MlpLayout& L, float* Y,
                       int64_t col_stride, int32_t* err, cudaStream_t s)
{
    static int attr_done[kMaxDevices] = {};  // per instantiation and device
    const int smem = (int)sizeof(TcSmem<NOUT>);
    cudaError_t e = smem_attr_per_device(k_mlp_forward_tc<NOUT>, smem, attr_done);
    if (e != cudaSuccess) return e;
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const int64_t tiles = (rows + kTcRows - 1) / kTcRows;
    int64_t blocks = sms;  // one block per SM: all 512 TMEM columns, four groups of 128 rows
    if (blocks > (tiles + kFwGroups - 1) / kFwGroups) blocks = (tiles + kFwGroups - 1) / kFwGroups;
    if (blocks < 1) return cudaSuccess;
    k_mlp_forward_tc<NOUT><<<(unsigned)blocks, kFwThreads, smem, s>>>(
        reinterpret_cast<const __nv_bfloat16*>(X), rows, reinterpret_cast<const unsigned char*>(params), L, Y, col_stride,
        err);
    return cudaGetLastError();
}

}  // namespace

cudaError_t mlp_forward_tc(const void* X, int64_t rows, const void* params, int K, float* Y, int32_t* err,
                           cudaStream_t s, int64_t col_stride)
{
    const MlpLayout L = mlp_layout(K);
    if (K == 16) return forward_tc<48>(X, rows, params, L, Y, col_stride, err, s);
    if (K == 8) return forward_tc<24>(X, rows, params, L, Y, col_stride, err, s);
    return cudaErrorInvalidValue;
}

}  // namespace lbt
