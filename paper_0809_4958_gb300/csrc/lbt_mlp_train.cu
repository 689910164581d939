// Training of the learned boundary upsampler: forward, loss, backward and Adam
// on the tcgen05 tensor cores (operand layout and helpers: lbt_tc.cuh).
//
// One kernel takes a 128-row tile from features and targets to its share of
// the gradient without leaving the SM: the activations, their gradients and
// the weights stay in shared memory, and every product of the backward pass
// reads them where they lie -- an operand stored for the forward product is
// its own transpose under an MN-major descriptor.  The weight gradients
// accumulate in TMEM over all tiles of a block and leave it once, as the
// block's partial; a second kernel adds the partials in a fixed order,
// applies Adam and writes the bf16 inference copy.
//
// What bounds it: latency.  A tile is a chain of six products, each an MMA, a
// commit, a wait and an epilogue, about 2 us in all, and the 16384 rows of the
// benchmark are 128 tiles, fewer than SMs; its 2.5 GFLOP would take 1.3 us and
// its bytes less.  One training step of 16384 rows (K = 16): 26.0 us, a sixth
// of it the reduction with Adam.  As a chain of twelve launches
// (forward, loss, three weight and two activation gradients that staged their
// operands transposed, three column sums, Adam, export) through global memory
// it took 240 us.  Eight warps, two to a TMEM quadrant, halve the epilogues.
#include <cuda_bf16.h>

#include "lbt_internal.h"
#include "lbt_tc.cuh"

namespace lbt {

namespace {

constexpr int kTrThreads = 256;  // eight warps: warps w and w + 4 read TMEM lanes 32 (w % 4) .. +31, each half of the columns
constexpr int kTrHalf = kMlpHidden / 2;
// TMEM columns
constexpr int kColWork = 0;      // Z1, Z2, Y, dH2, dH1 in turn
constexpr int kColW2 = 128;      // dW2 [in][out]
constexpr int kColW3 = 256;      // dW3 [hidden][out]
constexpr int kColW1 = 320;      // dW1, as [hidden][feature]
constexpr int kColB2 = 384;      // db2 in column 0
constexpr int kColB1 = 416;      // db1 in column 0
constexpr int kTrCols = 512;

template <int NOUT>
struct TrSmem {
    static constexpr int kNP = pad16(NOUT);
    __nv_bfloat16 w1[kMlpHidden * kMlpIn];
    __nv_bfloat16 w2[kMlpHidden * kMlpHidden];
    __nv_bfloat16 w3[kNP * kMlpHidden];
    __nv_bfloat16 x[kTcRows * kMlpIn];    // features with the ones of layer 1's bias in columns 24, 25
    __nv_bfloat16 xr[kTcRows * kMlpIn];   // features as given, for dW1
    __nv_bfloat16 h1[kTcRows * kMlpHidden];
    __nv_bfloat16 h2[kTcRows * kMlpHidden];   // then dZ1
    __nv_bfloat16 dz2[kTcRows * kMlpHidden];
    __nv_bfloat16 dy[kTcRows * kNP];
    __nv_bfloat16 ones[kTcRows * 16];
    __nv_bfloat16 bb2[kMlpHidden * 16];
    __nv_bfloat16 bb3[kNP * 16];
    float col[4][kNP];                    // column sums of dY by lane quadrant
    double loss[kTrThreads / 32];
    uint64_t bar;
    uint32_t tmem;
};
static_assert(sizeof(TrSmem<48>) <= 227 * 1024, "training shared memory");

// two adjacent gradients, kept where the activation is positive, as bf16
__device__ __forceinline__ uint32_t mask_pack(uint32_t h, uint32_t a, uint32_t b)
{
    const __nv_bfloat162 hb = *reinterpret_cast<const __nv_bfloat162*>(&h);
    const float x = __low2float(hb) > 0.f ? __uint_as_float(a) : 0.f;
    const float y = __high2float(hb) > 0.f ? __uint_as_float(b) : 0.f;
    const __nv_bfloat162 p = __floats2bfloat162_rn(x, y);
    return *reinterpret_cast<const uint32_t*>(&p);
}

// Columns [c0, c0 + 64) of this thread's accumulator row, masked by row m of
// the activation h, to row m of dst (both [128][128] operands; dst may be h).
__device__ __forceinline__ void masked_epilogue(uint32_t taddr, const __nv_bfloat16* h, __nv_bfloat16* dst, int m, int c0)
{
    uint32_t r[kTrHalf];
    tc_ld32_nowait(taddr, r);
    tc_ld32_nowait(taddr + 32, r + 32);
    tc_ld_wait();
#pragma unroll
    for (int g = 0; g < kTrHalf; g += 8) {
        const uint4 hv = *reinterpret_cast<const uint4*>(h + core_off(m, c0 + g, kMlpHidden));
        *reinterpret_cast<uint4*>(dst + core_off(m, c0 + g, kMlpHidden)) =
            make_uint4(mask_pack(hv.x, r[g], r[g + 1]), mask_pack(hv.y, r[g + 2], r[g + 3]),
                       mask_pack(hv.z, r[g + 4], r[g + 5]), mask_pack(hv.w, r[g + 6], r[g + 7]));
    }
}

// D += A B over NK steps of 16 along the reduction; a_step, b_step: bytes one
// step advances an operand.
template <int NK>
__device__ __forceinline__ void mma_chain(uint32_t d, uint32_t a, uint32_t a_step, uint32_t a_lbo, uint32_t a_sbo,
                                          uint32_t b, uint32_t b_step, uint32_t b_lbo, uint32_t b_sbo, uint32_t idesc,
                                          bool acc)
{
#pragma unroll
    for (int k = 0; k < NK; k++)
        tc_mma(d, tc_desc(a + k * a_step, a_lbo, a_sbo), tc_desc(b + k * b_step, b_lbo, b_sbo), idesc, acc || k > 0);
}

// partial: [gridDim.x][nmaster] gradient partials in master layout, loss_part
// and late [gridDim.x]: late is 1 where an MMA did not complete in time, and
// the partial is not to be used.  scale = 1 / (rows NOUT).
template <int NOUT>
__global__ void __launch_bounds__(kTrThreads, 1) k_mlp_train_tc(const __nv_bfloat16* __restrict__ X,
                                                                const float* __restrict__ T, int64_t rows,
                                                                const unsigned char* __restrict__ params, MlpLayout L,
                                                                float scale, float* __restrict__ partial,
                                                                double* __restrict__ loss_part, int* __restrict__ late)
{
    using Sm = TrSmem<NOUT>;
    constexpr int NP = Sm::kNP, OH = NP / 2;  // output columns of a thread
    extern __shared__ __align__(128) unsigned char tr_smem_raw[];
    Sm& sm = *reinterpret_cast<Sm*>(tr_smem_raw);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int q = warp & 3, half = warp >> 2;
    const int m = 32 * q + lane;  // row of the tile (and TMEM lane) this thread owns with its partner half

    stage_operand<kMlpHidden, kMlpIn>(sm.w1, reinterpret_cast<const __nv_bfloat16*>(params + L.w1), kMlpHidden, tid, kTrThreads);
    stage_operand<kMlpHidden, kMlpHidden>(sm.w2, reinterpret_cast<const __nv_bfloat16*>(params + L.w2), kMlpHidden, tid,
                                          kTrThreads);
    stage_operand<NP, kMlpHidden>(sm.w3, reinterpret_cast<const __nv_bfloat16*>(params + L.w3), NOUT, tid, kTrThreads);
    if (tid == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(su32(&sm.bar)) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(su32(&sm.tmem)),
                     "r"(kTrCols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    __syncthreads();  // W1 rows 24, 25 are overwritten below
    const float* b1 = reinterpret_cast<const float*>(params + L.b1);
    for (int n = tid; n < kMlpHidden; n += kTrThreads)
        split_bias(b1[n], sm.w1[core_off(n, kMlpFeat, kMlpIn)], sm.w1[core_off(n, kMlpFeat + 1, kMlpIn)]);
    stage_ones(sm.ones, tid, kTrThreads);
    stage_bias(sm.bb2, kMlpHidden, reinterpret_cast<const float*>(params + L.b2), kMlpHidden, tid, kTrThreads);
    stage_bias(sm.bb3, NP, reinterpret_cast<const float*>(params + L.b3), NOUT, tid, kTrThreads);

    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = sm.tmem;
    const uint32_t trow = tmem + ((uint32_t)(32 * q) << 16);
    const uint32_t work = tmem + kColWork;
    // byte offsets between core matrices of [.][32], [.][128], [.][NP] and [.][16] operands
    constexpr uint32_t kCore = 128, kR32 = (kMlpIn / 8) * 128, kR128 = (kMlpHidden / 8) * 128, kRNP = (NP / 8) * 128,
                       kR16 = 256;
    const uint32_t id_h = tc_idesc(kTcRows, kMlpHidden), id_o = tc_idesc(kTcRows, NP);
    const uint32_t ax = su32(sm.x), axr = su32(sm.xr), a1 = su32(sm.h1), a2 = su32(sm.h2), az2 = su32(sm.dz2),
                   ay = su32(sm.dy), aw1 = su32(sm.w1), aw2 = su32(sm.w2), aw3 = su32(sm.w3), aone = su32(sm.ones),
                   ab2 = su32(sm.bb2), ab3 = su32(sm.bb3);

    float colsum[OH];  // this thread's share of sum_r dY[r][o], FP32
#pragma unroll
    for (int c = 0; c < OH; c++) colsum[c] = 0.f;
    double sq = 0.0;  // sum of the squares of Y - T
    uint32_t phase = 0;
    bool ok = true, first = true;
    const bool t_vec = (reinterpret_cast<uintptr_t>(T) & 15) == 0;

    // Every thread's shared-memory writes visible to the tensor cores, then
    // one thread issues; and: wait for everything issued (false: the MMAs did
    // not complete within a second).
    auto issue_fence = [&]() {
        proxy_fence();
        tc_fence_before();
        __syncthreads();
        tc_fence_after();
    };
    auto wait_mma = [&]() {
        const bool arrived = tc_wait(&sm.bar, phase);
        phase ^= 1u;
        ok = __syncthreads_and(arrived);
        tc_fence_after();
        return ok;
    };

    float t[OH];  // targets, then Y - T
    // The squares of the row's differences, a share at a time: an FP64 instruction of a warp takes its quarter of the SM
    // 64 cycles, so the shares go where the block waits for an MMA anyway, the last one behind the next tile's (or the
    // partial's stores).  A step of 16384 / 65536 rows: 26.0 / 47.8 us; thirds widened by the conversion's rules, branch
    // by branch: 27.1 / 51.8; two FP32 words, which hold 48 bits: 24.6 / 41.0.
    constexpr int kShare = (OH + 3) / 4, kLast = OH - 3 * kShare;
    float dl[kLast > 0 ? kLast : 1];  // differences of the last share
#pragma unroll
    for (int c = 0; c < kLast; c++) dl[c] = 0.f;
    auto add_squares = [&](const float* d, int n) {
        bool plain = true;  // normal numbers and zeros
#pragma unroll
        for (int c = 0; c < kShare; c++)
            if (c < n) plain = plain && (d[c] == 0.f || (fabsf(d[c]) >= 1.17549435e-38f && fabsf(d[c]) <= 3.402823466e38f));
        if (plain) {
#pragma unroll
            for (int c = 0; c < kShare; c++)
                if (c < n) {
                    const uint32_t b = __float_as_uint(d[c]) & 0x7fffffffu;
                    const double x = __hiloint2double(b ? (int)((b >> 3) + 0x38000000u) : 0, (int)(b << 29));
                    sq = fma(x, x, sq);
                }
        } else {
#pragma unroll
            for (int c = 0; c < kShare; c++)
                if (c < n) sq = fma((double)d[c], (double)d[c], sq);
        }
    };

    const int64_t ntiles = (rows + kTcRows - 1) / kTcRows;
    for (int64_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
        const int64_t r = tile * kTcRows + m;
        const bool in = r < rows;
        // the row's features (half of them each) and targets
        {
            const uint4* src = reinterpret_cast<const uint4*>(X + (in ? r : 0) * kMlpIn) + 2 * half;
#pragma unroll
            for (int c = 0; c < 2; c++) {
                uint4 v = in ? __ldg(src + c) : make_uint4(0u, 0u, 0u, 0u);
                *reinterpret_cast<uint4*>(sm.xr + core_off(m, 8 * (2 * half + c), kMlpIn)) = v;
                if (2 * half + c == kMlpFeat / 8) v.x = 0x3F803F80u;  // bf16 1.0 twice
                *reinterpret_cast<uint4*>(sm.x + core_off(m, 8 * (2 * half + c), kMlpIn)) = v;
            }
        }
        {
            const float* tr = T + (in ? r : 0) * NOUT + half * OH;
#pragma unroll
            for (int c = 0; c < OH; c += 4) {
                const bool have = in && half * OH + c < NOUT;  // NOUT and OH are multiples of four
                if (t_vec) {
                    const float4 v = have ? __ldg(reinterpret_cast<const float4*>(tr + c)) : make_float4(0.f, 0.f, 0.f, 0.f);
                    t[c] = v.x;
                    t[c + 1] = v.y;
                    t[c + 2] = v.z;
                    t[c + 3] = v.w;
                } else {
                    for (int k = 0; k < 4; k++) t[c + k] = have ? __ldg(tr + c + k) : 0.f;
                }
            }
        }
        // forward: Z1, Z2, Y (the biases inside the MMAs)
        issue_fence();
        if (tid == 0) {
            mma_chain<kMlpIn / 16>(work, ax, 256, kCore, kR32, aw1, 256, kCore, kR32, id_h, false);
            tc_commit(&sm.bar);
        }
        if (!wait_mma()) break;
        {
            uint32_t v[kTrHalf];
            tc_ld32_nowait(trow + kColWork + half * kTrHalf, v);
            tc_ld32_nowait(trow + kColWork + half * kTrHalf + 32, v + 32);
            tc_ld_wait();
            relu_store<kTrHalf>(v, sm.h1, m, half * kTrHalf);
        }
        issue_fence();
        if (tid == 0) {
            mma_chain<kMlpHidden / 16>(work, a1, 256, kCore, kR128, aw2, 256, kCore, kR128, id_h, false);
            mma_chain<1>(work, aone, 0, kCore, kR16, ab2, 0, kCore, kR16, id_h, true);
            tc_commit(&sm.bar);
        }
        add_squares(dl, kLast);  // the tile before
        if (!wait_mma()) break;
        {
            uint32_t v[kTrHalf];
            tc_ld32_nowait(trow + kColWork + half * kTrHalf, v);
            tc_ld32_nowait(trow + kColWork + half * kTrHalf + 32, v + 32);
            tc_ld_wait();
            relu_store<kTrHalf>(v, sm.h2, m, half * kTrHalf);
        }
        issue_fence();
        if (tid == 0) {
            mma_chain<kMlpHidden / 16>(work, a2, 256, kCore, kR128, aw3, 256, kCore, kR128, id_o, false);
            mma_chain<1>(work, aone, 0, kCore, kR16, ab3, 0, kCore, kR16, id_o, true);
            tc_commit(&sm.bar);
        }
        if (!wait_mma()) break;
        // Y - T; dY = 2 (Y - T) scale, its column sums in FP32, itself in bf16 for the MMAs
        {
            uint32_t v[OH];
            tc_ld16_nowait(trow + kColWork + half * OH, v);
            if constexpr (OH == 24) tc_ld8_nowait(trow + kColWork + half * OH + 16, v + 16);
            tc_ld_wait();
            uint32_t pk[OH / 2];
#pragma unroll
            for (int c = 0; c < OH; c++) {
                t[c] = in && half * OH + c < NOUT ? __uint_as_float(v[c]) - t[c] : 0.f;
                colsum[c] += 2.f * t[c] * scale;
            }
#pragma unroll
            for (int c = 0; c < OH / 2; c++) {
                const __nv_bfloat162 p = __floats2bfloat162_rn(2.f * t[2 * c] * scale, 2.f * t[2 * c + 1] * scale);
                pk[c] = *reinterpret_cast<const uint32_t*>(&p);
            }
#pragma unroll
            for (int c = 0; c < OH; c += 8)
                *reinterpret_cast<uint4*>(sm.dy + core_off(m, half * OH + c, NP)) =
                    make_uint4(pk[c / 2], pk[c / 2 + 1], pk[c / 2 + 2], pk[c / 2 + 3]);
        }
        issue_fence();
        if (tid == 0) {
            // dH2 = dY W3^T: W3 [o][i] as the MN-major B [i][o]
            mma_chain<NP / 16>(work, ay, 256, kCore, kRNP, aw3, 2 * kR128, kR128, kCore,
                               tc_idesc(kTcRows, kMlpHidden, false, true), false);
            tc_commit(&sm.bar);
            // dW3 += H2^T dY, while the epilogue of dH2 runs
            mma_chain<kTcRows / 16>(tmem + kColW3, a2, 2 * kR128, kR128, kCore, ay, 2 * kRNP, kRNP, kCore,
                                    tc_idesc(kMlpHidden, NP, true, true), !first);
        }
        add_squares(t, kShare);
        if (!wait_mma()) break;
        masked_epilogue(trow + kColWork + half * kTrHalf, sm.h2, sm.dz2, m, half * kTrHalf);
        issue_fence();
        if (tid == 0) {
            // dH1 = dZ2 W2^T
            mma_chain<kMlpHidden / 16>(work, az2, 256, kCore, kR128, aw2, 2 * kR128, kR128, kCore,
                                       tc_idesc(kTcRows, kMlpHidden, false, true), false);
            tc_commit(&sm.bar);  // covers dW3 as well: H2 may be overwritten after the wait
            // dW2 += H1^T dZ2, db2 += dZ2^T 1
            mma_chain<kTcRows / 16>(tmem + kColW2, a1, 2 * kR128, kR128, kCore, az2, 2 * kR128, kR128, kCore,
                                    tc_idesc(kMlpHidden, kMlpHidden, true, true), !first);
            mma_chain<kTcRows / 16>(tmem + kColB2, az2, 2 * kR128, kR128, kCore, aone, 2 * kR16, kR16, kCore,
                                    tc_idesc(kMlpHidden, 16, true, true), !first);
        }
        add_squares(t + kShare, kShare);
        if (!wait_mma()) break;
        masked_epilogue(trow + kColWork + half * kTrHalf, sm.h1, sm.h2, m, half * kTrHalf);
        issue_fence();
        if (tid == 0) {
            // dW1^T += dZ1^T X, db1 += dZ1^T 1
            mma_chain<kTcRows / 16>(tmem + kColW1, a2, 2 * kR128, kR128, kCore, axr, 2 * kR32, kR32, kCore,
                                    tc_idesc(kMlpHidden, kMlpIn, true, true), !first);
            mma_chain<kTcRows / 16>(tmem + kColB1, a2, 2 * kR128, kR128, kCore, aone, 2 * kR16, kR16, kCore,
                                    tc_idesc(kMlpHidden, 16, true, true), !first);
            tc_commit(&sm.bar);
        }
        first = false;
        add_squares(t + 2 * kShare, kShare);
#pragma unroll
        for (int c = 0; c < kLast; c++) dl[c] = t[3 * kShare + c];
        if (!wait_mma()) break;  // every operand read: the next tile may be staged
    }
    if (!ok) tc_wait(&sm.bar, phase ^ 1u);  // let an MMA still in flight finish (bounded); `late` below says what happened

    // the block's partial in master layout; lane m is the row of each D
    float* P = partial + (int64_t)blockIdx.x * L.nmaster;
    {
        float* w2 = P + L.m_w2 + m * kMlpHidden + half * kTrHalf;
#pragma unroll 1
        for (int c0 = 0; c0 < kTrHalf; c0 += 32) {
            uint32_t v[32];
            tc_ld32_nowait(trow + kColW2 + half * kTrHalf + c0, v);
            tc_ld_wait();
#pragma unroll
            for (int c = 0; c < 32; c += 4) *reinterpret_cast<uint4*>(w2 + c0 + c) = make_uint4(v[c], v[c + 1], v[c + 2], v[c + 3]);
        }
        uint32_t v[OH];
        tc_ld16_nowait(trow + kColW3 + half * OH, v);
        if constexpr (OH == 24) tc_ld8_nowait(trow + kColW3 + half * OH + 16, v + 16);
        tc_ld_wait();
        float* w3 = P + L.m_w3 + m * NOUT + half * OH;
#pragma unroll
        for (int c = 0; c < OH; c += 4)
            if (half * OH + c < NOUT) *reinterpret_cast<uint4*>(w3 + c) = make_uint4(v[c], v[c + 1], v[c + 2], v[c + 3]);
        uint32_t w[16];
        tc_ld16_nowait(trow + kColW1 + half * 16, w);
        tc_ld_wait();
#pragma unroll
        for (int f = 0; f < 16; f++) P[L.m_w1 + (half * 16 + f) * kMlpHidden + m] = __uint_as_float(w[f]);
        tc_ld8_nowait(trow + (half ? kColB2 : kColB1), w);
        tc_ld_wait();
        P[(half ? L.m_b2 : L.m_b1) + m] = __uint_as_float(w[0]);
    }
    // column sums and loss over the block, in a fixed order
#pragma unroll
    for (int c = 0; c < OH; c++) {
        for (int o = 16; o > 0; o >>= 1) colsum[c] += __shfl_xor_sync(0xffffffffu, colsum[c], o);
        if (lane == 0) sm.col[q][half * OH + c] = colsum[c];
    }
    if (ok) add_squares(dl, kLast);
    double loss = sq;
    for (int o = 16; o > 0; o >>= 1) loss += __shfl_xor_sync(0xffffffffu, loss, o);
    if (lane == 0) sm.loss[warp] = loss;
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (tid < NOUT) P[L.m_b3 + tid] = (sm.col[0][tid] + sm.col[1][tid]) + (sm.col[2][tid] + sm.col[3][tid]);
    if (tid == 0) {
        double t = 0.0;
        for (int w = 0; w < kTrThreads / 32; w++) t += sm.loss[w];
        loss_part[blockIdx.x] = t * scale;
        late[blockIdx.x] = !ok;
    }
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTrCols) : "memory");
}

// Gradient = the blocks' partials added in a fixed order; then (ADAM) Adam on
// the master weights and the bf16 / FP32 inference copy of what changed.  A
// block takes 32 parameters (a lane each) in eight slices of the partials.
// Where a block's MMAs were late, gradient and loss are NaN and the weights and
// their moments stay as they are.
constexpr int kRdSlices = 8;
static_assert(kMlpMaxPartials <= 32 * kRdSlices, "a thread per block's flag");

struct AdamArgs {
    float *master, *m, *v;
    unsigned char* params;
    float lr, b1, b2, eps, c1, c2;
};

// element e of the master vector to its place in the inference parameters
__device__ __forceinline__ void export_one(int64_t e, float w, const MlpLayout& L, unsigned char* params)
{
    __nv_bfloat16* w1 = reinterpret_cast<__nv_bfloat16*>(params + L.w1);
    __nv_bfloat16* w2 = reinterpret_cast<__nv_bfloat16*>(params + L.w2);
    __nv_bfloat16* w3 = reinterpret_cast<__nv_bfloat16*>(params + L.w3);
    const int k = (int)e;
    if (k < L.m_b1) w1[(k % kMlpHidden) * kMlpIn + k / kMlpHidden] = __float2bfloat16_rn(w);
    else if (k < L.m_w2) reinterpret_cast<float*>(params + L.b1)[k - L.m_b1] = w;
    else if (k < L.m_b2) w2[((k - L.m_w2) % kMlpHidden) * kMlpHidden + (k - L.m_w2) / kMlpHidden] = __float2bfloat16_rn(w);
    else if (k < L.m_w3) reinterpret_cast<float*>(params + L.b2)[k - L.m_b2] = w;
    else if (k < L.m_b3) w3[((k - L.m_w3) % L.nout) * kMlpHidden + (k - L.m_w3) / L.nout] = __float2bfloat16_rn(w);
    else reinterpret_cast<float*>(params + L.b3)[k - L.m_b3] = w;
}

template <bool ADAM>
__global__ void __launch_bounds__(32 * kRdSlices) k_mlp_reduce(const float* __restrict__ partial,
                                                               const double* __restrict__ loss_part,
                                                               const int* __restrict__ late, int nparts, MlpLayout L, float* __restrict__ grad, float* grad_out,
                                                               double* loss, double* loss_out, AdamArgs A)
{
    __shared__ float sh[kRdSlices][32];
    const int lane = threadIdx.x & 31, slice = threadIdx.x >> 5;
    const int64_t e = (int64_t)blockIdx.x * 32 + lane;
    float acc = 0.f;
    if (e < L.nmaster)
#pragma unroll 8
        for (int p = slice; p < nparts; p += kRdSlices) acc += partial[(int64_t)p * L.nmaster + e];
    sh[slice][lane] = acc;
    const bool failed = __syncthreads_or((int)threadIdx.x < nparts && late[threadIdx.x] != 0);
    if (slice == 0 && e < L.nmaster) {
        float g = 0.f;
#pragma unroll
        for (int k = 0; k < kRdSlices; k++) g += sh[k][lane];
        if (failed) g = __int_as_float(0x7fc00000);
        grad[e] = g;
        if (grad_out) grad_out[e] = g;
        if (ADAM && !failed) {
            const float mi = A.b1 * A.m[e] + (1.f - A.b1) * g;
            const float vi = A.b2 * A.v[e] + (1.f - A.b2) * g * g;
            A.m[e] = mi;
            A.v[e] = vi;
            const float w = A.master[e] - A.lr * (mi / A.c1) / (sqrtf(vi / A.c2) + A.eps);
            A.master[e] = w;
            export_one(e, w, L, A.params);
        }
    }
    if (blockIdx.x == 0 && slice == 1) {  // the loss, by another warp of the first block
        double t = 0.0;
        for (int p = lane; p < nparts; p += 32) t += loss_part[p];
        for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
        if (failed) t = __longlong_as_double(0x7ff8000000000000ll);
        if (lane == 0) {
            *loss = t;
            if (loss_out) *loss_out = t;
        }
    }
}

__global__ void k_export(const float* master, MlpLayout L, unsigned char* params)
{
    const int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (e < L.nmaster) export_one(e, master[e], L, params);
}

template <int NOUT>
cudaError_t train_tc(const void* X, const float* T, int64_t rows, const unsigned char* params, const MlpLayout& L,
                     float* partial, double* loss_part, int* late, int blocks, cudaStream_t s)
{
    static int attr_done[kMaxDevices] = {};  // per instantiation and device
    const int smem = (int)sizeof(TrSmem<NOUT>);
    cudaError_t e = smem_attr_per_device(k_mlp_train_tc<NOUT>, smem, attr_done);
    if (e != cudaSuccess) return e;
    k_mlp_train_tc<NOUT><<<(unsigned)blocks, kTrThreads, smem, s>>>(reinterpret_cast<const __nv_bfloat16*>(X), T, rows,
                                                                    params, L, 1.0f / (float)(rows * L.nout), partial,
                                                                    loss_part, late);
    return cudaGetLastError();
}

}  // namespace

cudaError_t mlp_train(unsigned char* ws, const MlpTrain& W, const void* X, const float* T, int64_t rows, float* grad_out,
                      double* loss_out, bool adam, float lr, int64_t t, cudaStream_t s)
{
    float* f = reinterpret_cast<float*>(ws);
    unsigned char* params = ws + W.params_byte;
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    int64_t blocks = (rows + kTcRows - 1) / kTcRows;  // one tile a block up to the SMs (the workspace holds as many partials)
    if (blocks > sms) blocks = sms;
    if (blocks > kMlpMaxPartials) blocks = kMlpMaxPartials;
    double* loss_part = reinterpret_cast<double*>(f + W.loss_part);
    int* late = reinterpret_cast<int*>(f + W.late);
    cudaError_t e = W.K == 16 ? train_tc<48>(X, T, rows, params, W.L, f + W.partial, loss_part, late, (int)blocks, s)
                              : train_tc<24>(X, T, rows, params, W.L, f + W.partial, loss_part, late, (int)blocks, s);
    if (e != cudaSuccess) return e;
    const unsigned grid = (unsigned)((W.L.nmaster + 31) / 32);
    double* loss = reinterpret_cast<double*>(f + W.loss);
    AdamArgs A{};
    if (adam) {
        const float b1 = 0.9f, b2 = 0.999f;
        A = {f + W.master, f + W.m, f + W.v, params, lr, b1, b2, 1e-8f, 1.f - powf(b1, (float)t), 1.f - powf(b2, (float)t)};
        k_mlp_reduce<true><<<grid, 32 * kRdSlices, 0, s>>>(f + W.partial, loss_part, late, (int)blocks, W.L, f + W.grad,
                                                           grad_out, loss, loss_out, A);
    } else {
        k_mlp_reduce<false><<<grid, 32 * kRdSlices, 0, s>>>(f + W.partial, loss_part, late, (int)blocks, W.L, f + W.grad,
                                                            grad_out, loss, loss_out, A);
    }
    return cudaGetLastError();
}

cudaError_t mlp_export(const float* master, int K, void* params, cudaStream_t s)
{
    const MlpLayout L = mlp_layout(K);
    k_export<<<(unsigned)((L.nmaster + 255) / 256), 256, 0, s>>>(master, L, reinterpret_cast<unsigned char*>(params));
    return cudaGetLastError();
}

}  // namespace lbt
