// Stream-collide with the boundary layer, staged through shared memory by
// TMA bulk copies (cp.async.bulk) in a warp-specialised pipeline.
//
// A tile is kSites consecutive sites of one box.  For population i the sites
// of a tile pull from one contiguous source range shifted by c_iy E + c_iz E^2
// (and by c_ix inside the row), so one bulk copy per population, widened by a
// 16-byte halo on each side for the x shift, brings everything the tile needs
// into shared memory; the x shift becomes an offset into that row.
//
// One producer warp claims tiles from a global counter and issues their 19
// copies into a ring of stages; a "full" barrier per stage counts the bytes
// landing, an "empty" barrier counts the consumer warps done with the stage.
// Fifteen consumer warps take the stages in order.  A consumer warp loads its
// sites' populations from the stage into registers and releases the stage at
// once, then collides and stores straight to global memory, so the copies of
// a later tile into that stage overlap the arithmetic and the stores of this
// one.  No block-wide barrier is taken inside the loop.
//
// Only sites whose pull source crosses a periodic face (a wrap) read global
// memory directly.  Copies are clamped to the box's arrays; sites whose
// source lies outside are boundary sites, which are overwritten with the
// boundary equilibrium anyway.
#pragma once
#include <cstddef>

#include "lbt_device.cuh"
#include "lbt_fluct.cuh"

namespace lbt {

constexpr int kStagedHaloBytes = 16;  // x-shift halo on each side of a row
constexpr int kStagedConsumerWarps = 15;  // + the producer: four warps per scheduler
constexpr int kStagedConsumers = kStagedConsumerWarps * 32;
constexpr int kStagedThreads = kStagedConsumers + 32;  // + the producer warp
constexpr int kStagedHeaderBytes = 4096;               // barriers and tile headers
constexpr int kStagedMaxStages = 6;

// Tile geometry for SPT sites per consumer thread.  As many stages as fit in
// the 227 KB of shared memory a block may use (at most six).
template <int ST, int SPT>
struct Staged {
    using E = typename Stor<ST>::E;
    static constexpr int kSites = kStagedConsumers * SPT;
    static constexpr int kRowBytes = kSites * (int)sizeof(E);               // one population row of a tile
    static constexpr int kRowStride = kRowBytes + 2 * kStagedHaloBytes;
    static constexpr int kStageBytes = kQ * kRowStride;
    static constexpr int kFit = (227 * 1024 - kStagedHeaderBytes) / kStageBytes;
    static constexpr int kStages = kFit > kStagedMaxStages ? kStagedMaxStages : kFit;
    // what is left of the shared memory holds the x-face boundary samples of
    // each stage's rows (the paired bodies; see stage_edges)
    static constexpr bool kEdges = SPT == 2 && ST != kF64;
    static constexpr int kEdgeBytes =
        kEdges ? (227 * 1024 - kStagedHeaderBytes - kStages * kStageBytes) / kStages / 16 * 16 : 0;
    static constexpr int kSmemBytes = kStagedHeaderBytes + kStages * (kStageBytes + kEdgeBytes);
    static constexpr int kHalo = kStagedHaloBytes / (int)sizeof(E);         // halo elements
    static_assert(kStages >= 2, "tile too large for a two-stage pipeline");
    static_assert(kRowStride % 16 == 0, "bulk copies need 16-byte aligned rows");
};

// Sites per consumer thread the staged kernel supports per storage format
// (the first is the default): FP64 1; FP32 2 or 1; 16-bit 2 or 1.
inline bool staged_spt_ok(int storage, int spt) { return spt == 1 || (spt == 2 && storage != kF64); }
inline int staged_default_spt(int storage) { return storage == kF64 ? 1 : 2; }
inline int staged_tile_sites(int spt) { return kStagedConsumers * spt; }

// ---- PTX helpers (mbarrier + bulk copy) ----
__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}

__device__ __forceinline__ void fence_mbar_init() { asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory"); }

__device__ __forceinline__ void fence_proxy_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

__device__ __forceinline__ void mbar_arrive(uint64_t* bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}

__device__ __forceinline__ void mbar_arrive_expect_tx(uint64_t* bar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}

__device__ __forceinline__ void bulk_load(void* dst, const void* src, uint32_t bytes, uint64_t* bar)
{
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                     smem_u32(dst)),
                 "l"(src), "r"(bytes), "r"(smem_u32(bar))
                 : "memory");
}

// The populations stream through L2 once per step (both buffers together
// exceed it): their stores, and with chains in the launch (SCParams::
// hint_loads) also the bulk copies of the pulled rows, go in with the
// evict-first policy, so that what is reused -- the boundary sample ring, box
// records, the bead kernel's code and data -- stays in L2.  (Measured: the
// evict-first loads make the chain-free 256^3 sweep slower, the 128^3 step
// with its bead kernel faster.)
constexpr bool kL2HintStores = true;

__device__ __forceinline__ uint64_t l2_evict_first_policy()
{
    uint64_t pol;
    asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(pol));
    return pol;
}

__device__ __forceinline__ void bulk_load_hint(void* dst, const void* src, uint32_t bytes, uint64_t* bar, uint64_t pol)
{
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1], %2, [%3], %4;" ::"r"(
            smem_u32(dst)),
        "l"(src), "r"(bytes), "r"(smem_u32(bar)), "l"(pol)
        : "memory");
}

// Store of one population value or pair, evict-first when the hints are on.
template <class T>
__device__ __forceinline__ void st_stream(T* p, T v)
{
    if constexpr (kL2HintStores) __stcs(p, v);
    else *p = v;
}

// Test the phase; a thread that finds it incomplete may be suspended in
// hardware for up to 20 us (or until the phase completes) instead of spinning
// and taking issue slots from the warps that compute.
__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t phase)
{
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\tselp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(phase), "r"(20000u)
        : "memory");
    return ok != 0;
}

__device__ __forceinline__ uint64_t global_ns()
{
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// Wait for a phase of the barrier, giving up after limit_ns nanoseconds (one
// second by default; shorter only when a test makes a wait run out on purpose).
__device__ __forceinline__ bool mbar_wait_bounded(uint64_t* bar, uint32_t phase, int64_t limit_ns)
{
    if (mbar_try_wait(bar, phase)) return true;
    const uint64_t t0 = global_ns();
    while (!mbar_try_wait(bar, phase))
        if (global_ns() - t0 > (uint64_t)limit_ns) return false;
    return true;
}

// Box of tile t (the largest b with tile_prefix[b] <= t), searched by a whole
// warp: 32 candidates per round, so 512 boxes take two dependent loads.
__device__ __forceinline__ int locate_box_warp(const SCParams& p, int64_t t, int lane)
{
    int lo = 0, hi = p.nboxes - 1;
    while (lo < hi) {
        const int step = (hi - lo + 32) / 32;
        const int idx = lo + lane * step;
        const bool le = idx <= hi && p.tile_prefix[idx] <= t;
        const unsigned m = __ballot_sync(0xffffffffu, le);  // a prefix of the lanes; lane 0 always (prefix[lo] <= t)
        lo += (31 - __clz(m)) * step;
        hi = min(hi, lo + step - 1);
    }
    return lo;
}

// Shared-memory header: full and empty barriers, then the tile header the
// producer writes for each stage before it arms the barrier: the box record,
// first site, frozen flag, and what the collision and the boundary layer of
// the box need at this step -- BGK constants in the arithmetic type, the ring
// slots and weights of the time interpolation, the upsampler substep -- so
// that they are worked out (64-bit divisions, FP64 conversions, global loads)
// once per tile by the producer, not once per consumer warp.
template <int ST>
struct StagedTile {
    using A = typename Stor<ST>::A;
    using R = typename Stor<ST>::R;
    BoxDev bd;
    int64_t s0;
    int64_t step;  // the step n -> n + 1 of the launch
    int32_t box;
    int32_t mlp_s;
    int32_t frozen;  // the box carries an error status: its state does not change
    int32_t slot[4];
    R c[4];
    A om, om1, srcfac, drho_b;  // 1/tau, 1 - 1/tau, 1 - 1/(2 tau), rho_b - 1
    A acc[3], pad;              // body acceleration of the step
    // x-face samples of the tile's rows in the stage (edge_stride 0: not
    // staged): edge_n samples of weight edge_c, then the upsampler residual
    int32_t edge_row, edge_stride, edge_n, edge_mlp;
    R edge_c[4];
};
// Consumers keep reading a tile's header after they have released its data
// stage (early release), so headers live in a ring of twice the stages: tile
// k uses header k mod 2S, which the producer rewrites for tile k + 2S only
// after every consumer warp has released tile k + S -- that is, after each of
// them has finished tile k (a warp takes the tiles in order).
template <int ST>
struct StagedHeader {
    uint64_t full[kStagedMaxStages];
    uint64_t empty[kStagedMaxStages];
    StagedTile<ST> t[2 * kStagedMaxStages];
};
static_assert(sizeof(StagedHeader<kF64>) <= kStagedHeaderBytes, "header does not fit");
static_assert(sizeof(StagedHeader<kF32>) <= kStagedHeaderBytes, "header does not fit");

// Quotient and remainder of a site index by E with a precomputed multiplier:
// q = (s * m) >> 40 with m = ceil(2^40 / E), exact for s < 2^31 and E <= 1024.
__device__ __forceinline__ int div_e(int64_t s, uint64_t m) { return (int)(((uint64_t)s * m) >> 40); }

// One site per consumer thread (FP64, and the reduced formats with one site a
// thread): thread c (0 .. 479) takes site s0 + c, so the lanes of a warp read
// consecutive shared-memory words and store consecutive global words.  The
// site's populations go to registers, the warp releases the stage, then the
// collision (BGK by opposite pairs, whose equilibrium has an even part in
// common and an odd part that changes sign) and the stores.  FP64 is bound by
// its arithmetic (two lanes a clock on an SM), so its instructions are counted:
// about 125 a site in place of 212 (each population's momentum and relaxation
// by itself, a division), 128^3 in 544 us in place of 713.
template <int ST, bool PER, bool ACCEL>
__device__ __forceinline__ void staged_tile(const SCParams& p, const StagedTile<ST>& th, const unsigned char* stage,
                                            uint64_t* empty)
{
    using S = Stor<ST>;
    using E = typename S::E;
    using A = typename S::A;
    using R = typename S::R;
    constexpr int H = Staged<ST, 1>::kHalo;
    const int tid = threadIdx.x;
    // site indices of a box fit 32 bits (E <= 1024)
    const int s = (int)th.s0 + tid;
    const BoxDev& bd = th.bd;
    const int Ei = bd.E;
    const int n3 = (int)bd.n3;
    const int per = bd.per_mask;
    const bool px = per & 1, py = per & 2, pz = per & 4;
    const E* Ab = reinterpret_cast<const E*>(p.A) + bd.f_off;
    E* Bb = reinterpret_cast<E*>(p.B) + bd.f_off;

    const bool act = s < n3;
    const int row = div_e(act ? s : 0, bd.div_magic);
    const int x = (act ? s : 0) - row * Ei;
    const int z = div_e(row, bd.div_magic);
    const int y = row - z * Ei;
    const bool bnd = act && ((!px && (x == 0 || x == Ei - 1)) || (!py && (y == 0 || y == Ei - 1)) ||
                             (!pz && (z == 0 || z == Ei - 1)));

    // f_i pulled into the site: shared memory, or global memory across a
    // periodic wrap; zero where it is not used (boundary and inactive sites)
    A f[kQ];
#pragma unroll
    for (int i = 0; i < kQ; i++) {
        const int cx = cvec(i, 0), cy = cvec(i, 1), cz = cvec(i, 2);
        A v = S::in(reinterpret_cast<const E*>(stage + i * Staged<ST, 1>::kRowStride)[H + tid - cx]);
        if (PER) {
            const int xs = x - cx, ys = y - cy, zs = z - cz;
            const bool wrap = (px && (xs < 0 || xs >= Ei)) || (py && (ys < 0 || ys >= Ei)) ||
                              (pz && (zs < 0 || zs >= Ei));
            if (wrap && act)
                v = S::in(Ab[(int64_t)i * n3 + ((int64_t)wrapi(zs, Ei) * Ei + wrapi(ys, Ei)) * Ei + wrapi(xs, Ei)]);
        }
        f[i] = act && !bnd ? v : A(0);
    }
    __syncwarp();
    if ((tid & 31) == 0) mbar_arrive(empty);  // this warp is done with the stage

    A r = f[0], j[3];
#pragma unroll
    for (int i = 1; i < kQ; i += 2) {
        const A d = f[i] - f[i + 1];
        r += f[i] + f[i + 1];
#pragma unroll
        for (int c = 0; c < 3; c++) {
            if (i == 1 + 2 * c) j[c] = d;  // the axis pairs come first
            else if (cvec(i, c) > 0) j[c] += d;
            else if (cvec(i, c) < 0) j[c] -= d;
        }
    }
    A rho = A(1) + r;
    // flag the box (it freezes from the next step on) where a collided site's
    // density is not finite or not positive; NaN fails both comparisons
    const bool nonfinite = !(rho > A(0) && rho < A(1e30));
    if (__any_sync(0xffffffffu, nonfinite) && (tid & 31) == 0) atomicCAS(&p.status[th.box], 0, LB_ERR_NONFINITE);
    A ac[3] = {A(0), A(0), A(0)};
    if (ACCEL)
        for (int c = 0; c < 3; c++) {
            ac[c] = th.acc[c];
            j[c] += A(0.5) * rho * ac[c];
        }
    const A inv = site_inverse(rho);
    A ux = j[0] * inv, uy = j[1] * inv, uz = j[2] * inv;
    A om = th.om, om1 = th.om1, sf = th.srcfac;
    // boundary sites: equilibrium of the boundary velocity from the ring
    if (bnd) {
        TimeWeights<R> tw;
#pragma unroll
        for (int a = 0; a < 4; a++) {
            tw.slot[a] = th.slot[a];
            tw.c[a] = th.c[a];
        }
        int pp, qq;
        const int fc = owning_face(x, y, z, Ei, per, pp, qq);
        float res[3];
        load_mlp_residual(p, bd, th.mlp_s, fc, pp, qq, res);
        R ub[3];
        boundary_velocity<R>(reinterpret_cast<const R*>(p.ring), p.ring_slot_elems, bd, fc, pp, qq, tw, ub);
        add_mlp_residual<R>(p, bd, res, ub);
        r = th.drho_b;
        rho = A(1) + r;
        ux = (A)ub[0];
        uy = (A)ub[1];
        uz = (A)ub[2];
        om = A(1);
        om1 = sf = A(0);
    }
    const A xx = ux * ux, yy = uy * uy, zz = uz * uz;
    // with k = om w rho, w = 1/18: om times the equilibrium of a pair is
    // (w om drho - k 1.5 u^2) + k 4.5 cu^2 +- k 3 cu on an axis, half that on an edge
    const A om18 = A(1) / A(18) * om, k18 = om18 * rho;
    const A b18 = om18 * r - k18 * (A(1.5) * (xx + yy + zz)), b36 = A(0.5) * b18;
    const A q18 = A(4.5) * k18, q36 = A(2.25) * k18, t18 = A(3) * k18, t36 = A(1.5) * k18;
    A s18 = A(0), s36 = A(0), ua3 = A(0);
    if (ACCEL) {
        s18 = A(1) / A(18) * sf * rho;
        s36 = A(0.5) * s18;
        ua3 = A(-3) * (ux * ac[0] + uy * ac[1] + uz * ac[2]);
    }
    // populations are written in order 0, 1, ..., 18 through one running pointer
    E* out = Bb + s;
    {
        A val = om1 * f[0] + A(6) * b18;
        if (ACCEL) val += A(6) * s18 * ua3;
        if (act) st_stream(out, S::out(val));
    }
#pragma unroll
    for (int i = 1; i < kQ; i += 2) {
        out += i == 1 ? n3 : 2 * n3;  // row of population i; population i + 1 is one row further
        const int cx = cvec(i, 0), cy = cvec(i, 1), cz = cvec(i, 2);
        const bool axis = i < 7;
        // c_i . u of the first of the pair (an axis pair starts with the positive
        // direction, an edge pair with its first component positive)
        const A first = cx ? ux : (cy ? uy : uz), second = cz ? uz : uy;
        const A cu = axis ? first : ((cx ? (cy ? cy : cz) : cz) > 0 ? first + second : first - second);
        const A cu2 = axis ? (cx ? xx : (cy ? yy : zz)) : cu * cu;
        A even = (axis ? q18 : q36) * cu2 + (axis ? b18 : b36);
        A plus = even + (axis ? t18 : t36) * cu, minus = even - (axis ? t18 : t36) * cu;
        if (ACCEL) {
            A ca = A(0);  // c_i . a; c -> -c flips c.a and c.u
            if (cx) ca += cx * ac[0];
            if (cy) ca += cy * ac[1];
            if (cz) ca += cz * ac[2];
            const A sw = axis ? s18 : s36, e = A(9) * ca * cu + ua3;
            plus += sw * (e + A(3) * ca);
            minus += sw * (e - A(3) * ca);
        }
        if (act) {
            st_stream(out, S::out(om1 * f[i] + plus));
            st_stream(out + n3, S::out(om1 * f[i + 1] + minus));
        }
    }
}

// ---- two adjacent sites per consumer thread (FP32 and 16-bit storage) -----
// Packed FP32 arithmetic: one instruction advances both sites of a thread.
__device__ __forceinline__ float2 f2(float a) { return make_float2(a, a); }
__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }
// a - b as one packed FMA: b (-1) is exact, so this is a - b rounded once
__device__ __forceinline__ float2 sub2(float2 a, float2 b) { return __ffma2_rn(b, make_float2(-1.f, -1.f), a); }
__device__ __forceinline__ float2 mul2(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }

// Loads and stores of a pair of adjacent stored elements: one aligned word
// for the pair of a thread (elements e, e + 1 with e even), two scalar loads
// for the x-shifted pairs, conversions to and from FP32 packed where the
// format has a packed instruction (round to nearest even, as Stor<ST>::out).
template <int ST>
struct PairIO;
template <>
struct PairIO<kF32> {
    using E = float;
    static __device__ __forceinline__ float2 even(const E* row, int e) { return *reinterpret_cast<const float2*>(row + e); }
    static __device__ __forceinline__ float2 any(const E* row, int e) { return make_float2(row[e], row[e + 1]); }
    static __device__ __forceinline__ void store(E* p, float2 v) { st_stream(reinterpret_cast<float2*>(p), v); }
};
template <>
struct PairIO<kF16> {
    using E = uint16_t;
    static __device__ __forceinline__ float2 even(const E* row, int e)
    {
        return __half22float2(*reinterpret_cast<const __half2*>(row + e));
    }
    static __device__ __forceinline__ float2 any(const E* row, int e)
    {
        return make_float2(__half2float(__ushort_as_half(row[e])), __half2float(__ushort_as_half(row[e + 1])));
    }
    static __device__ __forceinline__ void store(E* p, float2 v)
    {
        const __half2 h = __floats2half2_rn(v.x, v.y);
        st_stream(reinterpret_cast<unsigned int*>(p), *reinterpret_cast<const unsigned int*>(&h));
    }
};
template <>
struct PairIO<kBF16> {
    using E = uint16_t;
    static __device__ __forceinline__ float2 even(const E* row, int e)
    {
        return __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(row + e));
    }
    static __device__ __forceinline__ float2 any(const E* row, int e)
    {
        return make_float2(__bfloat162float(__ushort_as_bfloat16(row[e])),
                           __bfloat162float(__ushort_as_bfloat16(row[e + 1])));
    }
    static __device__ __forceinline__ void store(E* p, float2 v)
    {
        const __nv_bfloat162 h = __floats2bfloat162_rn(v.x, v.y);
        st_stream(reinterpret_cast<unsigned int*>(p), *reinterpret_cast<const unsigned int*>(&h));
    }
};

// Boundary velocity of the two adjacent sites x, x + 1 (x even) of a row on
// face f (a y or z face, in-face row q): eight-byte loads, the arithmetic of
// boundary_velocity and add_mlp_residual.
template <int ST>
__device__ __forceinline__ void boundary_velocity_pair(const SCParams& p, const StagedTile<ST>& th, int f, int q, int x,
                                                       float2 u[3])
{
    const BoxDev& bd = th.bd;
    const int64_t fe = (int64_t)bd.E * bd.E;
    const float* ring = reinterpret_cast<const float*>(p.ring) + bd.ring_off + (3 * f) * fe + (int64_t)q * bd.E + x;
#pragma unroll
    for (int c = 0; c < 3; c++) {
        u[c] = f2(0.f);
#pragma unroll
        for (int a = 0; a < 4; a++)
            if (th.c[a] != 0.f)  // a zero weight never touches its (possibly unpushed) slot
                u[c] = fma2(f2(th.c[a]), __ldg(reinterpret_cast<const float2*>(ring + (int64_t)th.slot[a] * p.ring_slot_elems + c * fe)),
                            u[c]);
    }
    if (bd.mlp_row >= 0) {
        const float* y = p.mlp_y + (int64_t)(3 * (th.mlp_s - 1)) * p.mlp_ystride + bd.mlp_row + f * fe + (int64_t)q * bd.E + x;
#pragma unroll
        for (int c = 0; c < 3; c++)
            u[c] = fma2(f2(p.mlp_yunit), __ldg(reinterpret_cast<const float2*>(y + c * p.mlp_ystride)), u[c]);
    }
}

// Boundary velocity of a site on x face f (0 or 1) in box row `row` from the
// samples staged with the tile.
template <int ST>
__device__ __forceinline__ void edge_velocity(const SCParams& p, const StagedTile<ST>& th, const float* edge, int f,
                                              int row, float u[3])
{
    const int st = th.edge_stride;
    const float* e = edge + 3 * f * st + (row - th.edge_row);
#pragma unroll
    for (int c = 0; c < 3; c++) u[c] = 0.f;
    for (int a = 0; a < th.edge_n; a++, e += 6 * st)
#pragma unroll
        for (int c = 0; c < 3; c++) u[c] += th.edge_c[a] * e[c * st];
    if (th.edge_mlp)
#pragma unroll
        for (int c = 0; c < 3; c++) u[c] += p.mlp_yunit * e[c * st];
}

// Velocity and density deviation of the boundary sites among a thread's
// adjacent pair (x, x + 1) of box row `row` = (y, z): ue is the x-face site's
// velocity where the tile's samples were staged (staged), else it is loaded here.
template <int ST>
__device__ __forceinline__ void boundary_pair(const SCParams& p, const StagedTile<ST>& th, int row, int x, int y, int z,
                                              bool brow, bool xface0, bool xface1, bool staged, float ue[3], float2& ux,
                                              float2& uy, float2& uz, float2& drho)
{
    const BoxDev& bd = th.bd;
    const int Ei = bd.E;
    const bool py = bd.per_mask & 2;
    if (brow) {  // a row on a y or z face (its x-face sites, which belong to the x faces, follow)
        const int f = !py && y == 0 ? 2 : (!py && y == Ei - 1 ? 3 : (z == 0 ? 4 : 5));
        float2 u[3];
        boundary_velocity_pair(p, th, f, f < 4 ? z : y, x, u);
        ux = u[0];
        uy = u[1];
        uz = u[2];
        drho = f2(th.drho_b);
    }
    if (xface0 || xface1) {
        if (!staged) {
            TimeWeights<float> tw;
#pragma unroll
            for (int a = 0; a < 4; a++) {
                tw.slot[a] = th.slot[a];
                tw.c[a] = th.c[a];
            }
            float res[3];
            load_mlp_residual(p, bd, th.mlp_s, xface1, y, z, res);
            boundary_velocity<float>(reinterpret_cast<const float*>(p.ring), p.ring_slot_elems, bd, xface1, y, z, tw, ue);
            add_mlp_residual<float>(p, bd, res, ue);
        }
        if (xface0) {
            drho.x = th.drho_b;
            ux.x = ue[0];
            uy.x = ue[1];
            uz.x = ue[2];
        } else {
            drho.y = th.drho_b;
            ux.y = ue[0];
            uy.y = ue[1];
            uz.y = ue[2];
        }
    }
}

// Consumer thread c (0 .. 479) of one tile of 960 sites takes the adjacent
// sites s0 + 2c and s0 + 2c + 1 (same row: E and s0 are even), so a warp
// reads and writes 64 consecutive sites with one word per lane.  Same
// arithmetic as staged_tile, on both sites at once; a boundary site takes
// om = 1, 1 - om = 0 and no force term in its lane, which turns the
// collision into its equilibrium.
template <int ST, bool PER, bool ACCEL>
__device__ __forceinline__ void staged_tile_pair(const SCParams& p, const StagedTile<ST>& th, const unsigned char* stage,
                                                 uint64_t* empty)
{
    static_assert(ST != kF64, "the paired body works in FP32");
    using S = Stor<ST>;
    using E = typename S::E;
    using IO = PairIO<ST>;
    constexpr int H = Staged<ST, 2>::kHalo;
    const int tid = threadIdx.x;
    const int s0 = (int)th.s0;
    const BoxDev& bd = th.bd;
    const int Ei = bd.E;
    const int n3 = (int)bd.n3;
    const int per = bd.per_mask;
    const bool px = per & 1, py = per & 2, pz = per & 4;
    const E* Ab = reinterpret_cast<const E*>(p.A) + bd.f_off;
    E* Bb = reinterpret_cast<E*>(p.B) + bd.f_off;

    const int s = s0 + 2 * tid;  // first site of the pair (even)
    const bool act = s < n3;     // n3 is even: both sites or none
    const int row = div_e(act ? s : 0, bd.div_magic);
    const int x = (act ? s : 0) - row * Ei;
    const int z = div_e(row, bd.div_magic);
    const int y = row - z * Ei;
    const bool brow = act && ((!py && (y == 0 || y == Ei - 1)) || (!pz && (z == 0 || z == Ei - 1)));
    const bool xface0 = act && !px && x == 0, xface1 = act && !px && x + 1 == Ei - 1;  // never both: E >= 8
    const bool bnd0 = brow || xface0, bnd1 = brow || xface1;
    const bool keep0 = act && !bnd0, keep1 = act && !bnd1;

    // f_i pulled into both sites (zero where unused)
    float2 f[kQ];
#pragma unroll
    for (int i = 0; i < kQ; i++) {
        const int cx = cvec(i, 0), cy = cvec(i, 1), cz = cvec(i, 2);
        const E* row = reinterpret_cast<const E*>(stage + i * Staged<ST, 2>::kRowStride);
        float2 v = cx == 0 ? IO::even(row, H + 2 * tid) : IO::any(row, H + 2 * tid - cx);
        if (PER) {
            const int ys = y - cy, zs = z - cz;
            const bool wyz = (py && (ys < 0 || ys >= Ei)) || (pz && (zs < 0 || zs >= Ei));
#pragma unroll
            for (int k = 0; k < 2; k++) {
                const int xs = x + k - cx;
                const bool wrap = wyz || (px && (xs < 0 || xs >= Ei));
                if (wrap && act) {
                    const float w = S::in(
                        Ab[(int64_t)i * n3 + ((int64_t)wrapi(zs, Ei) * Ei + wrapi(ys, Ei)) * Ei + wrapi(xs, Ei)]);
                    if (k == 0) v.x = w;
                    else v.y = w;
                }
            }
        }
        // boundary lanes keep what they pulled (finite: the stage holds copied
        // or zeroed elements only); it is multiplied by zero below
        f[i] = v;
    }
    // x-face velocity: staged with the tile (read before the stage is released)
    float ue[3];
    const bool staged_edges = th.edge_stride != 0;
    if ((xface0 || xface1) && staged_edges)
        edge_velocity(p, th, reinterpret_cast<const float*>(stage + Staged<ST, 2>::kStageBytes), xface1, row, ue);
    __syncwarp();
    if ((tid & 31) == 0) mbar_arrive(empty);  // this warp is done with the stage

    // moments (sum of deviations, momentum)
    float2 r = f[0];
#pragma unroll
    for (int i = 1; i < kQ; i++) r = add2(r, f[i]);
    float2 jx = sub2(f[1], f[2]), jy = sub2(f[3], f[4]), jz = sub2(f[5], f[6]);
    jx = add2(jx, sub2(f[7], f[8]));
    jy = add2(jy, sub2(f[7], f[8]));
    jx = add2(jx, sub2(f[9], f[10]));
    jy = sub2(jy, sub2(f[9], f[10]));
    jx = add2(jx, sub2(f[11], f[12]));
    jz = add2(jz, sub2(f[11], f[12]));
    jx = add2(jx, sub2(f[13], f[14]));
    jz = sub2(jz, sub2(f[13], f[14]));
    jy = add2(jy, sub2(f[15], f[16]));
    jz = add2(jz, sub2(f[15], f[16]));
    jy = add2(jy, sub2(f[17], f[18]));
    jz = sub2(jz, sub2(f[17], f[18]));
    float2 rho = add2(f2(1.f), r);
    const bool nonfinite = (keep0 && !(rho.x > 0.f && rho.x < 1e30f)) || (keep1 && !(rho.y > 0.f && rho.y < 1e30f));
    if (__any_sync(0xffffffffu, nonfinite) && (tid & 31) == 0) atomicCAS(&p.status[th.box], 0, LB_ERR_NONFINITE);
    float2 ac[3] = {f2(0.f), f2(0.f), f2(0.f)};
    if (ACCEL) {
        for (int c = 0; c < 3; c++) ac[c] = f2(th.acc[c]);
        const float2 hr = mul2(f2(0.5f), rho);
        jx = fma2(hr, ac[0], jx);
        jy = fma2(hr, ac[1], jy);
        jz = fma2(hr, ac[2], jz);
    }
    // 1 / rho by the fast reciprocal (within 2 ulp; the FP32 collision rounds
    // O(1) terms at 2^-24 anyway)
    const float2 inv = make_float2(__fdividef(1.f, rho.x), __fdividef(1.f, rho.y));
    float2 ux = mul2(jx, inv), uy = mul2(jy, inv), uz = mul2(jz, inv);
    float2 drho = r;

    // boundary sites: equilibrium of the boundary velocity from the ring
    if (bnd0 || bnd1) {
        boundary_pair(p, th, row, x, y, z, brow, xface0, xface1, staged_edges, ue, ux, uy, uz, drho);
        rho = add2(f2(1.f), drho);
    }

    // per-lane relaxation: boundary lanes take their equilibrium
    const float2 om = make_float2(bnd0 ? 1.f : th.om, bnd1 ? 1.f : th.om);
    const float2 om1 = make_float2(bnd0 ? 0.f : th.om1, bnd1 ? 0.f : th.om1);
    const float2 usq = mul2(f2(1.5f), fma2(ux, ux, fma2(uy, uy, mul2(uz, uz))));
    const float2 nusq = mul2(f2(-1.f), usq);
    // om w rho and om w drho for the two weight classes of the moving
    // populations and the rest population; om 3 w rho for the odd part
    const float2 omrho = mul2(om, rho), omdrho = mul2(om, drho);
    const float2 r18 = mul2(f2(1.f / 18.f), omrho), d18 = mul2(f2(1.f / 18.f), omdrho);
    const float2 r36 = mul2(f2(1.f / 36.f), omrho), d36 = mul2(f2(1.f / 36.f), omdrho);
    const float2 t18 = mul2(f2(3.f / 18.f), omrho), t36 = mul2(f2(3.f / 36.f), omrho);
    float2 sfr, srcw[2], ua;
    if (ACCEL) {  // Guo source: (1 - om/2) w rho (3 (c.a - u.a) + 9 (c.u)(c.a)), zero on boundary lanes
        const float2 sf = make_float2(bnd0 ? 0.f : th.srcfac, bnd1 ? 0.f : th.srcfac);
        sfr = mul2(sf, rho);
        srcw[0] = mul2(sfr, f2(1.f / 18.f));
        srcw[1] = mul2(sfr, f2(1.f / 36.f));
        ua = fma2(ux, ac[0], fma2(uy, ac[1], mul2(uz, ac[2])));
    }
    E* out = Bb + s;
    // population 0: om w0 (drho - rho usq)
    {
        const float2 odeq = mul2(f2(1.f / 3.f), fma2(omrho, nusq, omdrho));
        float2 val = fma2(om1, f[0], odeq);
        if (ACCEL) val = fma2(sfr, make_float2(-ua.x, -ua.y), val);  // (1 - om/2) w0 rho 3 (-u.a), 3 w0 = 1
        if (act) IO::store(out, val);
    }
#pragma unroll
    for (int i = 1; i < kQ; i += 2) {
        out += i == 1 ? n3 : 2 * n3;  // row of population i; population i + 1 is one row further
        const int cx = cvec(i, 0), cy = cvec(i, 1), cz = cvec(i, 2);
        const bool w18 = i < 7;
        float2 cu;
        if (cx && cy) cu = cy > 0 ? (cx > 0 ? add2(ux, uy) : make_float2(-(ux.x + uy.x), -(ux.y + uy.y))) : (cx > 0 ? sub2(ux, uy) : sub2(uy, ux));
        else if (cx && cz) cu = cz > 0 ? (cx > 0 ? add2(ux, uz) : make_float2(-(ux.x + uz.x), -(ux.y + uz.y))) : (cx > 0 ? sub2(ux, uz) : sub2(uz, ux));
        else if (cy && cz) cu = cz > 0 ? (cy > 0 ? add2(uy, uz) : make_float2(-(uy.x + uz.x), -(uy.y + uz.y))) : (cy > 0 ? sub2(uy, uz) : sub2(uz, uy));
        else cu = cx ? ux : (cy ? uy : uz);  // axis pairs: c_i = +x, +y or +z for odd i
        // om (w (drho + rho (4.5 cu^2 - usq))) and om (3 w rho cu)
        const float2 t = fma2(mul2(f2(4.5f), cu), cu, nusq);
        const float2 oeven = fma2(w18 ? r18 : r36, t, w18 ? d18 : d36);
        const float2 oodd = mul2(w18 ? t18 : t36, cu);
        float2 vp = fma2(om1, f[i], add2(oeven, oodd));
        float2 vm = fma2(om1, f[i + 1], sub2(oeven, oodd));
        if (ACCEL) {
            float ca = 0.f;  // c_i . a (uniform per box)
            if (cx) ca += cx * ac[0].x;
            if (cy) ca += cy * ac[1].x;
            if (cz) ca += cz * ac[2].x;
            const float2 sw = w18 ? srcw[0] : srcw[1];
            // + : 3 (ca - ua) + 9 cu ca ;  - : 3 (-ca - ua) + 9 cu ca  (c -> -c flips ca and cu)
            const float2 nine_cu_ca = mul2(f2(9.f * ca), cu);
            const float2 sp = fma2(f2(3.f), sub2(f2(ca), ua), nine_cu_ca);
            const float2 sm = fma2(f2(3.f), sub2(f2(-ca), ua), nine_cu_ca);
            vp = fma2(sw, sp, vp);
            vm = fma2(sw, sm, vm);
        }
        if (act) {
            IO::store(out, vp);
            IO::store(out + n3, vm);
        }
    }
}

// Consumer body of a box with the fluctuating collision (lbt_fluct.cuh), one
// site a thread (FP64, and the reduced formats with one site a thread): the
// site pulled into registers, the stage released, then the moments and either
// the boundary equilibrium or the fluctuating collision with the site's Philox
// noise of step n.  Boxes with a body force or a chain do not take this path.
template <int ST, bool PER>
__device__ __forceinline__ void staged_tile_fluct(const SCParams& p, const StagedTile<ST>& th,
                                                  const unsigned char* stage, uint64_t* empty, int64_t n)
{
    using S = Stor<ST>;
    using E = typename S::E;
    using A = typename S::A;
    using R = typename S::R;
    constexpr int H = Staged<ST, 1>::kHalo;
    const int tid = threadIdx.x;
    const int s = (int)th.s0 + tid;
    const BoxDev& bd = th.bd;
    const int Ei = bd.E;
    const int n3 = (int)bd.n3;
    const int per = bd.per_mask;
    const bool px = per & 1, py = per & 2, pz = per & 4;
    const E* Ab = reinterpret_cast<const E*>(p.A) + bd.f_off;
    E* Bb = reinterpret_cast<E*>(p.B) + bd.f_off;

    const bool act = s < n3;
    const int row = div_e(act ? s : 0, bd.div_magic);
    const int x = (act ? s : 0) - row * Ei;
    const int z = div_e(row, bd.div_magic);
    const int y = row - z * Ei;
    const bool bnd = act && ((!px && (x == 0 || x == Ei - 1)) || (!py && (y == 0 || y == Ei - 1)) ||
                             (!pz && (z == 0 || z == Ei - 1)));
    A d[kQ], r = A(0), j[3] = {A(0), A(0), A(0)};
#pragma unroll
    for (int i = 0; i < kQ; i++) {
        const int cx = cvec(i, 0), cy = cvec(i, 1), cz = cvec(i, 2);
        A v = S::in(reinterpret_cast<const E*>(stage + i * Staged<ST, 1>::kRowStride)[H + tid - cx]);
        if (PER) {
            const int xs = x - cx, ys = y - cy, zs = z - cz;
            const bool wrap = (px && (xs < 0 || xs >= Ei)) || (py && (ys < 0 || ys >= Ei)) ||
                              (pz && (zs < 0 || zs >= Ei));
            if (wrap && act)
                v = S::in(Ab[(int64_t)i * n3 + ((int64_t)wrapi(zs, Ei) * Ei + wrapi(ys, Ei)) * Ei + wrapi(xs, Ei)]);
        }
        d[i] = act && !bnd ? v : A(0);
        r += d[i];
#pragma unroll
        for (int c = 0; c < 3; c++)
            if (cvec(i, c)) j[c] += cvec(i, c) * d[i];
    }
    __syncwarp();
    if ((tid & 31) == 0) mbar_arrive(empty);  // this warp is done with the stage

    const A rho = A(1) + r;
    const bool nonfinite = !(rho > A(0) && rho < A(1e30));
    A out[kQ];
    if (bnd) {  // boundary equilibrium of the boundary velocity, as in the BGK bodies
        TimeWeights<R> tw;
#pragma unroll
        for (int a = 0; a < 4; a++) {
            tw.slot[a] = th.slot[a];
            tw.c[a] = th.c[a];
        }
        int pp, qq;
        const int fc = owning_face(x, y, z, Ei, per, pp, qq);
        float res[3];
        load_mlp_residual(p, bd, th.mlp_s, fc, pp, qq, res);
        R ub[3];
        boundary_velocity<R>(reinterpret_cast<const R*>(p.ring), p.ring_slot_elems, bd, fc, pp, qq, tw, ub);
        add_mlp_residual<R>(p, bd, res, ub);
        const A dr = th.drho_b, rb = A(1) + dr;
        const A u0 = (A)ub[0], u1 = (A)ub[1], u2 = (A)ub[2];
        const A usq = A(1.5) * (u0 * u0 + u1 * u1 + u2 * u2);
#pragma unroll
        for (int i = 0; i < kQ; i++) out[i] = fluct_deq<A>(i, dr, rb, u0, u1, u2, usq);
    } else {
        const A inv = A(1) / rho;
        fluct_collide<A>(d, r, j[0] * inv, j[1] * inv, j[2] * inv, p.fluct[th.box], n, s, out);
    }
    if (act)
#pragma unroll
        for (int i = 0; i < kQ; i++) Bb[(int64_t)i * n3 + s] = S::out(out[i]);
    if (__any_sync(0xffffffffu, nonfinite) && (tid & 31) == 0) atomicCAS(&p.status[th.box], 0, LB_ERR_NONFINITE);
}

// The fluctuating collision of two adjacent sites per thread (FP32 and 16-bit
// storage), in packed FP32.  An even mode sees only the sum of an opposite pair
// of populations, an odd one only the difference, so the two transforms come
// down to about a hundred additions for both sites together; the relaxation
// factors and noise amplitudes are read in FP32, folded with the mode norms.
// Arithmetic bound (the transforms, eight Philox calls a thread): 96^3 FP32 in
// 53.9 us a step; with 19 x 15 scalar transforms a site, the parameters
// converted from FP64 for every site and four-byte stores two sites apart, 109.
template <int ST, bool PER>
__device__ __forceinline__ void staged_tile_fluct_pair(const SCParams& p, const StagedTile<ST>& th,
                                                       const unsigned char* stage, uint64_t* empty, int64_t n)
{
    static_assert(ST != kF64, "the paired body works in FP32");
    using S = Stor<ST>;
    using E = typename S::E;
    using IO = PairIO<ST>;
    constexpr int H = Staged<ST, 2>::kHalo;
    const int tid = threadIdx.x;
    const BoxDev& bd = th.bd;
    const int Ei = bd.E;
    const int n3 = (int)bd.n3;
    const int per = bd.per_mask;
    const bool px = per & 1, py = per & 2, pz = per & 4;
    const E* Ab = reinterpret_cast<const E*>(p.A) + bd.f_off;
    const int s = (int)th.s0 + 2 * tid;  // first site of the pair (even)
    const bool act = s < n3;             // n3 is even: both sites or none
    const int row = div_e(act ? s : 0, bd.div_magic);
    const int x = (act ? s : 0) - row * Ei;
    const int z = div_e(row, bd.div_magic);
    const int y = row - z * Ei;
    const bool brow = act && ((!py && (y == 0 || y == Ei - 1)) || (!pz && (z == 0 || z == Ei - 1)));
    const bool xface0 = act && !px && x == 0, xface1 = act && !px && x + 1 == Ei - 1;
    const bool bnd0 = brow || xface0, bnd1 = brow || xface1;

    float2 f[kQ];
#pragma unroll
    for (int i = 0; i < kQ; i++) {
        const int cx = cvec(i, 0), cy = cvec(i, 1), cz = cvec(i, 2);
        const E* src = reinterpret_cast<const E*>(stage + i * Staged<ST, 2>::kRowStride);
        float2 v = cx == 0 ? IO::even(src, H + 2 * tid) : IO::any(src, H + 2 * tid - cx);
        if (PER) {
            const int ys = y - cy, zs = z - cz;
            const bool wyz = (py && (ys < 0 || ys >= Ei)) || (pz && (zs < 0 || zs >= Ei));
#pragma unroll
            for (int k = 0; k < 2; k++) {
                const int xs = x + k - cx;
                if ((wyz || (px && (xs < 0 || xs >= Ei))) && act) {
                    const float w = S::in(
                        Ab[(int64_t)i * n3 + ((int64_t)wrapi(zs, Ei) * Ei + wrapi(ys, Ei)) * Ei + wrapi(xs, Ei)]);
                    if (k == 0) v.x = w;
                    else v.y = w;
                }
            }
        }
        f[i] = v;  // boundary lanes: not used
    }
    __syncwarp();
    if ((tid & 31) == 0) mbar_arrive(empty);  // this warp is done with the stage

    // opposite pairs: sums in f[i], differences in f[i + 1] (i odd)
    float2 r = f[0], j[3];
#pragma unroll
    for (int i = 1; i < kQ; i += 2) {
        const float2 a = f[i], b = f[i + 1];
        f[i] = add2(a, b);
        f[i + 1] = sub2(a, b);
        r = add2(r, f[i]);
#pragma unroll
        for (int c = 0; c < 3; c++) {
            if (i == 1 + 2 * c) j[c] = f[i + 1];  // the axis pairs come first
            else if (cvec(i, c) > 0) j[c] = add2(j[c], f[i + 1]);
            else if (cvec(i, c) < 0) j[c] = sub2(j[c], f[i + 1]);
        }
    }
    float2 rho = add2(f2(1.f), r);
    const bool nonfinite = (act && !bnd0 && !(rho.x > 0.f && rho.x < 1e30f)) || (act && !bnd1 && !(rho.y > 0.f && rho.y < 1e30f));
    if (__any_sync(0xffffffffu, nonfinite) && (tid & 31) == 0) atomicCAS(&p.status[th.box], 0, LB_ERR_NONFINITE);
    // 1 / rho to half an ulp (one Newton step on the hardware's approximation):
    // its error goes straight into the momentum the equilibrium carries
    float2 inv = make_float2(fast_inverse(rho.x), fast_inverse(rho.y));
    inv = fma2(inv, fma2(mul2(f2(-1.f), rho), inv, f2(1.f)), inv);
    float2 ux = mul2(j[0], inv), uy = mul2(j[1], inv), uz = mul2(j[2], inv), drho = r;
    const float2 srho = make_float2(sqrtf(rho.x), sqrtf(rho.y));
    if (bnd0 || bnd1) {
        float ue[3];
        boundary_pair(p, th, row, x, y, z, brow, xface0, xface1, false, ue, ux, uy, uz, drho);
        rho = add2(f2(1.f), drho);
    }
    // equilibrium of a pair: even part q cu^2 + b, odd part t cu
    const float2 xx = mul2(ux, ux), yy = mul2(uy, uy), zz = mul2(uz, uz);
    const float2 base = fma2(rho, mul2(f2(-1.5f), add2(xx, add2(yy, zz))), drho);
    // (the FP32 value of 1/18 is 7e-9 off, that of 1/6 3e-8: the momentum a step
    // carries over would grow by as much every step)
    const float2 k18 = mul2(f2(1.f / 18.f), rho);
    const float2 b18 = mul2(f2(1.f / 18.f), base), b36 = mul2(f2(0.5f), b18);
    const float2 q18 = mul2(f2(4.5f), k18), q36 = mul2(f2(2.25f), k18);
    const float2 t18 = mul2(f2(3.f), k18), t36 = mul2(f2(1.5f), k18);
    auto equilibrium = [&](int i, float2& even, float2& odd) {
        const int cx = cvec(i, 0), cy = cvec(i, 1), cz = cvec(i, 2);
        const bool axis = i < 7;
        const float2 first = cx ? ux : (cy ? uy : uz), second = cz ? uz : uy;
        const float2 cu = axis ? first : ((cx ? (cy ? cy : cz) : cz) > 0 ? add2(first, second) : sub2(first, second));
        even = fma2(axis ? q18 : q36, axis ? (cx ? xx : (cy ? yy : zz)) : mul2(cu, cu), axis ? b18 : b36);
        odd = mul2(axis ? t18 : t36, cu);
    };
    // non-equilibrium sums and differences, then the moments of modes 4 .. 18 (lbt_fluct.cuh)
    const float2 n0 = fma2(f2(-6.f), b18, f[0]);
#pragma unroll
    for (int i = 1; i < kQ; i += 2) {
        float2 even, odd;
        equilibrium(i, even, odd);
        f[i] = fma2(f2(-2.f), even, f[i]);
        f[i + 1] = fma2(f2(-2.f), odd, f[i + 1]);
    }
    float2 m[15];
    {
        const float2 exy = add2(f[7], f[9]), exz = add2(f[11], f[13]), eyz = add2(f[15], f[17]);
        const float2 es = add2(add2(exy, exz), eyz), as = add2(add2(f[1], f[3]), f[5]);
        m[0] = sub2(es, n0);
        m[12] = add2(fma2(f2(-2.f), as, es), n0);
        const float2 ax = fma2(f2(3.f), f[1], mul2(f2(-1.f), as)), ex = fma2(f2(-3.f), eyz, es);
        m[1] = add2(ax, ex);
        m[13] = sub2(ex, ax);
        const float2 ay = sub2(f[3], f[5]), ey = sub2(exy, exz);
        m[2] = add2(ay, ey);
        m[14] = sub2(ey, ay);
        m[3] = sub2(f[7], f[9]);
        m[4] = sub2(f[15], f[17]);
        m[5] = sub2(f[11], f[13]);
        const float2 sx = add2(f[8], f[10]), tx = add2(f[12], f[14]);
        m[6] = fma2(f2(-2.f), f[2], add2(sx, tx));
        m[9] = sub2(sx, tx);
        const float2 sy = sub2(f[8], f[10]), ty = add2(f[16], f[18]);
        m[7] = fma2(f2(-2.f), f[4], add2(sy, ty));
        m[10] = sub2(ty, sy);
        const float2 sz = sub2(f[12], f[14]), tz = sub2(f[16], f[18]);
        m[8] = fma2(f2(-2.f), f[6], add2(sz, tz));
        m[11] = sub2(sz, tz);
    }
    // relaxed moments plus noise, over their norms; none on boundary sites (selected, not multiplied by zero: what a
    // boundary site pulled means nothing, its density may have no square root and its values may be infinite)
    const FluctDev& fd = p.fluct[th.box];
    const uint32_t k0 = (uint32_t)fd.seed, k1 = (uint32_t)(fd.seed >> 32);
#pragma unroll
    for (int blk = 0; blk < 4; blk++) {
        uint32_t xa[4] = {(uint32_t)n, (uint32_t)s, (uint32_t)blk, 0xF1u}, xb[4] = {(uint32_t)n, (uint32_t)s + 1, (uint32_t)blk, 0xF1u};
        philox4x32_10(xa, k0, k1);
        philox4x32_10(xb, k0, k1);
        const float4 g = __ldg(reinterpret_cast<const float4*>(fd.gamma_f) + blk);
        const float4 a = __ldg(reinterpret_cast<const float4*>(fd.amp_f) + blk);
        const float gk[4] = {g.x, g.y, g.z, g.w}, ak[4] = {a.x, a.y, a.z, a.w};
#pragma unroll
        for (int w = 0; w < 4; w++)
            if (4 * blk + w < 15) {
                const float2 xi = make_float2(unit_uniform_t<float>(xa[w]), unit_uniform_t<float>(xb[w]));
                float2& mk = m[4 * blk + w];
                const float2 relaxed = fma2(f2(gk[w]), mk, mul2(mul2(f2(ak[w]), srho), xi));
                mk = make_float2(bnd0 ? 0.f : relaxed.x, bnd1 ? 0.f : relaxed.y);
            }
    }
    // back to the populations: equilibrium + w (even part +- odd part)
    E* out = reinterpret_cast<E*>(p.B) + bd.f_off + s;
    if (act) IO::store(out, fma2(f2(6.f), b18, mul2(f2(1.f / 3.f), sub2(m[12], m[0]))));
    const float2 G = add2(m[0], m[12]), Hh = add2(m[1], m[13]), I = add2(m[2], m[14]);
    const float2 h = sub2(m[1], m[13]), v = sub2(m[2], m[14]), c2 = mul2(f2(-2.f), m[12]);
#pragma unroll
    for (int i = 1; i < kQ; i += 2) {
        out += i == 1 ? n3 : 2 * n3;  // row of population i; population i + 1 is one row further
        float2 even, odd, e, o;
        equilibrium(i, even, odd);
        if (i == 1) e = fma2(f2(2.f), h, c2);
        else if (i == 3) e = add2(sub2(v, h), c2);
        else if (i == 5) e = sub2(sub2(c2, h), v);
        else if (i < 11) e = i == 7 ? add2(add2(add2(G, Hh), I), m[3]) : sub2(add2(add2(G, Hh), I), m[3]);
        else if (i < 15) e = i == 11 ? add2(sub2(add2(G, Hh), I), m[5]) : sub2(sub2(add2(G, Hh), I), m[5]);
        else e = i == 15 ? add2(fma2(f2(-2.f), Hh, G), m[4]) : sub2(fma2(f2(-2.f), Hh, G), m[4]);
        if (i < 7) o = mul2(f2(-2.f), m[6 + i / 2]);
        else if (i < 11) o = i == 7 ? add2(add2(m[6], m[9]), sub2(m[7], m[10])) : sub2(add2(m[6], m[9]), sub2(m[7], m[10]));
        else if (i < 15) o = i == 11 ? add2(sub2(m[6], m[9]), add2(m[8], m[11])) : sub2(sub2(m[6], m[9]), add2(m[8], m[11]));
        else o = i == 15 ? add2(add2(m[7], m[10]), sub2(m[8], m[11])) : sub2(add2(m[7], m[10]), sub2(m[8], m[11]));
        const float2 w = f2(i < 7 ? 1.f / 18.f : 1.f / 36.f);
        even = fma2(w, e, even);
        odd = fma2(w, o, odd);
        if (act) {
            IO::store(out, add2(even, odd));
            IO::store(out + n3, sub2(even, odd));
        }
    }
}

// Consumer warps: take the stages in order until the producer posts the end.
// KIND 0: every box of the launch is non-periodic and force-free, so only
// that tile body is compiled in (fewer registers than the kernel that carries
// all bodies).
template <int ST, int SPT, int KIND>
__device__ __forceinline__ void staged_consume(const SCParams& p, unsigned char* smem, StagedHeader<ST>* hd)
{
    constexpr bool GENERAL = KIND > 0;
    using G = Staged<ST, SPT>;
    using E = typename Stor<ST>::E;
    for (int k = 0;; k++) {
        const int st = k % G::kStages;
        const uint32_t phase = (uint32_t)((k / G::kStages) & 1);
        const bool arrived = mbar_wait_bounded(&hd->full[st], phase, p.wait_ns);
        if (!__all_sync(0xffffffffu, arrived)) {
            // nothing arrived within the limit: flag the box, let copies still
            // in flight land (one more bounded wait) and leave
            if ((threadIdx.x & 31) == 0) {
                const int b = *reinterpret_cast<volatile const int32_t*>(&hd->t[k % (2 * G::kStages)].box);
                atomicCAS(&p.status[b >= 0 && b < p.nboxes ? b : 0], 0, LB_ERR_TIMEOUT);
            }
            mbar_wait_bounded(&hd->full[st], phase, p.wait_ns);
            return;
        }
        const StagedTile<ST>& th = hd->t[k % (2 * G::kStages)];
        const int b = th.box;
        if (b < 0) return;  // end of work
        const int64_t s0 = th.s0;
        const BoxDev& bd = th.bd;
        const unsigned char* stage = smem + kStagedHeaderBytes + st * (G::kStageBytes + G::kEdgeBytes);
        if (th.frozen) {
            // frozen box: release the stage, the state does not change
            __syncwarp();
            if ((threadIdx.x & 31) == 0) mbar_arrive(&hd->empty[st]);
            const E* Ab = reinterpret_cast<const E*>(p.A) + bd.f_off;
            E* Bb = reinterpret_cast<E*>(p.B) + bd.f_off;
            for (int t = threadIdx.x; t < G::kSites; t += kStagedConsumers)
                if (s0 + t < bd.n3)
                    for (int i = 0; i < kQ; i++) Bb[(int64_t)i * bd.n3 + s0 + t] = Ab[(int64_t)i * bd.n3 + s0 + t];
        } else if (KIND == 2 && bd.fluct) {
            if constexpr (KIND == 2) {
                if constexpr (SPT == 2 && ST != kF64) {
                    if (bd.per_mask) staged_tile_fluct_pair<ST, true>(p, th, stage, &hd->empty[st], th.step);
                    else staged_tile_fluct_pair<ST, false>(p, th, stage, &hd->empty[st], th.step);
                } else {
                    if (bd.per_mask) staged_tile_fluct<ST, true>(p, th, stage, &hd->empty[st], th.step);
                    else staged_tile_fluct<ST, false>(p, th, stage, &hd->empty[st], th.step);
                }
            }
        } else if constexpr (SPT == 2 && ST != kF64) {  // adjacent site pairs, packed FP32
            if (!GENERAL) {
                staged_tile_pair<ST, false, false>(p, th, stage, &hd->empty[st]);
            } else if (bd.per_mask == 0) {
                if (bd.has_accel) staged_tile_pair<ST, false, true>(p, th, stage, &hd->empty[st]);
                else staged_tile_pair<ST, false, false>(p, th, stage, &hd->empty[st]);
            } else {
                if (bd.has_accel) staged_tile_pair<ST, true, true>(p, th, stage, &hd->empty[st]);
                else staged_tile_pair<ST, true, false>(p, th, stage, &hd->empty[st]);
            }
        } else if (!GENERAL) {
            staged_tile<ST, false, false>(p, th, stage, &hd->empty[st]);
        } else if (bd.per_mask == 0) {
            if (bd.has_accel) staged_tile<ST, false, true>(p, th, stage, &hd->empty[st]);
            else staged_tile<ST, false, false>(p, th, stage, &hd->empty[st]);
        } else {
            if (bd.has_accel) staged_tile<ST, true, true>(p, th, stage, &hd->empty[st]);
            else staged_tile<ST, true, false>(p, th, stage, &hd->empty[st]);
        }
    }
}

// Prefetch into L2 (evict-last) of the upsampler residuals of substep ms for
// the boundary sites of the box rows that tile [s0, s0 + T) covers: the
// x-face sites at both ends of every row (faces 0 and 1, in-face (y, z);
// staged: not those, they come with the tile) and whole rows on a y or z face,
// three components each.  One row per lane;
// every address lies inside the box's residual columns.
__device__ __forceinline__ void prefetch_l2(const float* a)
{
    asm volatile("prefetch.global.L2::evict_last [%0];" ::"l"(a));
}
__device__ __forceinline__ void prefetch_mlp_residuals(const SCParams& p, const BoxDev& bd, int ms, int64_t s0, int T,
                                                       int lane, bool staged)
{
    const int Eb = bd.E;
    const int64_t fe = (int64_t)Eb * Eb, str = p.mlp_ystride;
    const float* y0 = p.mlp_y + (int64_t)(3 * (ms - 1)) * str + bd.mlp_row;
    const int64_t r_first = s0 / Eb, r_end = (s0 + T - 1) / Eb + 1;
    for (int64_t r = r_first + lane; r < r_end && r < fe; r += 32) {
        const int yy = (int)(r % Eb), zz = (int)(r / Eb);
        if (!staged)
#pragma unroll
            for (int c = 0; c < 3; c++) {
                prefetch_l2(y0 + c * str + (int64_t)zz * Eb + yy);       // x- face
                prefetch_l2(y0 + c * str + fe + (int64_t)zz * Eb + yy);  // x+ face
            }
        const int fo = yy == 0 ? 2 : (yy == Eb - 1 ? 3 : (zz == 0 ? 4 : (zz == Eb - 1 ? 5 : -1)));
        if (fo >= 0) {
            const int q = fo < 4 ? zz : yy;  // in-face (x, z) on a y face, (x, y) on a z face
            const float* row = y0 + fo * fe + (int64_t)q * Eb;
            for (int x0 = 0; x0 < Eb; x0 += 32)
#pragma unroll
                for (int c = 0; c < 3; c++) prefetch_l2(row + c * str + x0);
        }
    }
}

// The samples of the x faces (sites x = 0 and E - 1) of the box rows a tile
// covers.  In a face sample [3][z][y] row (y, z) of the box is element z E + y,
// so the tile's rows are one run per face, component and sample: one bulk copy
// each, next to the tile's populations, in place of the loads from global
// memory that every warp with the end of a row waited for.  Lane k takes
// sample k / 6 of those with a weight, then the upsampler's residuals of the
// substep; face (k % 6) / 3, component k % 3.  Runs are `stride` elements long,
// start at a multiple of four (16 bytes) and lie inside E^2, itself a multiple
// of 64.  Fills the header's fields; returns the run's base (null: none),
// E^2 - stride in last_start.
//
// Boxes whose runs do not fit the room of a stage load from global memory.  In
// FP32 (2544 bytes) two samples, linear in time, fit from E = 24 on, Hermite's
// four from 48, and with the upsampler's residual from 64 (2400 bytes there,
// 2880 at 56); in 16-bit storage (960 bytes) two samples fit from 64, four, also
// with the residual, from 240.  Staged against loaded, us a step: FP32 linear 128
// boxes of 64^3 747 / 798, 512 of 32^3 418 / 453, one of 128^3 53.4 / 54.2; with the
// upsampler 128 of 64^3 849 / 889; binary16 linear 128 of 64^3 528 / 537, one of
// 256^3, where one site in 128 is on an x face, 232 / 224.
template <int ROOM, int ST>
__device__ __forceinline__ const float* edge_runs(const SCParams& p, StagedTile<ST>& th, int T, int lane, int& last_start)
{
    const BoxDev& bd = th.bd;
    const int fe = bd.E * bd.E;
    const int stride = ((T + bd.E - 2) / bd.E + 1 + 3 + 3) & ~3;  // rows a tile may touch, from a multiple of four
    int ns = 0, my_slot = 0;
    float my_c = 0.f;
#pragma unroll
    for (int a = 0; a < 4; a++)
        if (th.c[a] != 0.f) {  // a zero weight never touches its (possibly unpushed) slot
            if (lane / 6 == ns) my_slot = th.slot[a];
            if (lane == ns) my_c = th.c[a];
            ns++;
        }
    const bool mlp = bd.mlp_row >= 0;
    const int runs = 6 * (ns + (mlp ? 1 : 0));
    const bool fits = !(bd.per_mask & 1) && !bd.fluct && runs <= 32 && runs * stride * 4 <= ROOM && stride <= fe;
    if (lane < 4) th.edge_c[lane] = my_c;
    if (lane == 0) {
        th.edge_stride = fits ? stride : 0;
        th.edge_n = ns;
        th.edge_mlp = mlp;
    }
    last_start = fe - stride;
    if (!fits || lane >= runs) return nullptr;
    const int k = lane % 6;
    return lane < 6 * ns ? reinterpret_cast<const float*>(p.ring) + (int64_t)my_slot * p.ring_slot_elems + bd.ring_off +
                               (int64_t)k * fe
                         : p.mlp_y + (int64_t)(3 * (th.mlp_s - 1) + k % 3) * p.mlp_ystride + bd.mlp_row + (int64_t)(k / 3) * fe;
}

// Producer warp (the last warp): claims tiles from the global counter (reset
// to zero at the end of every step, so a block that starts late -- its SM
// still busy with the bead kernel -- simply takes fewer tiles) and fills the
// stages as the consumers free them.  Lane 0 claims and waits for the stage;
// lane i < 19 handles population row i: its source range, the zeroing of the
// part of the row that lies outside the box's arrays (those sites are boundary
// sites: their pulled values are multiplied by zero and must be finite, so no
// consumer may read what a previous tile left there), and its bulk copy.
//
// One tile's pass through this loop must stay below what the consumers take
// for a tile (2.2 us at 256^3 in 16-bit storage), or the copies starve.  The
// header and everything that depends on the box alone is therefore worked out
// when the box changes (records, status and samples from global memory, a few
// round trips) and kept in registers, the header as words spread over the
// lanes; a further tile of the box only stores them.  Launches with many tiles
// to a block claim several neighbours at once for the same reason.  (Worked out
// for every tile, 256^3 binary16 took 268 us a step and takes 220, 128^3 FP32
// under a body force 71.6 and 58.7; one more round trip a tile made them 330
// and 83.)
template <int ST, int SPT, int KIND>
__device__ __forceinline__ void staged_produce(const SCParams& p, unsigned char* smem, StagedHeader<ST>* hd)
{
    using G = Staged<ST, SPT>;
    using E = typename Stor<ST>::E;
    using R = typename Stor<ST>::R;
    using A = typename Stor<ST>::A;
    using Tile = StagedTile<ST>;
    constexpr int T = G::kSites, H = G::kHalo, W = T + 2 * H;
    constexpr int kWords = (int)(sizeof(Tile) / 8), kMine = (kWords + 31) / 32;  // header words, of one lane
    static_assert(sizeof(Tile) % 8 == 0 && offsetof(Tile, s0) % 8 == 0 && offsetof(Tile, bd) == 0, "header copied by words");
    static_assert(sizeof(BoxDev) % 8 == 0 && sizeof(BoxDev) / 8 <= 32, "box record copied by one warp");
    const int lane = threadIdx.x & 31;
    int cy = 0, cz = 0;  // y and z components of this lane's population
#pragma unroll
    for (int i = 0; i < kQ; i++)
        if (lane == i) {
            cy = cvec(i, 1);
            cz = cvec(i, 2);
        }
    const uint64_t pol = p.hint_loads ? l2_evict_first_policy() : 0;
    unsigned long long* ctr = reinterpret_cast<unsigned long long*>(p.tile_counter);
    const int run = p.claim;  // neighbouring tiles of one claim
    // the first claim of a block is fixed, the counter deals out the rest
    const long long dealt = (long long)gridDim.x * run;
    long long next = (long long)blockIdx.x * run;
    int left = run;  // tiles of the claim not yet taken
    // the record of an only box (written by nothing but copies between launches)
    const bool only = p.nboxes == 1;
    uint64_t only_word = 0;
    if (only && lane < (int)(sizeof(BoxDev) / 8)) only_word = reinterpret_cast<const uint64_t*>(p.boxes)[lane];
    // Launched as a programmatic dependent of the kernel before it on the
    // stream (the previous step's last): everything up to here may run while
    // that kernel does.  Wait for it to complete and its writes to be visible.
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const int64_t n = *p.step;
    const bool back = (n & 1) && p.withhold_tile < 0;
    // of the current box
    int64_t tile_lo = 0, tile_hi = 0;  // its tiles
    uint64_t hw[kMine];
    const E* row_src = nullptr;        // this lane's population, at its pull shift
    int64_t n3 = 0;
    int Ei = 1, fe = 1, shift = 0;
    uint64_t div_magic = 0;
    const float* edge_src = nullptr;
    int edge_bytes = 0, edge_last = 0, ms = 0;
    bool mlp = false;
    for (int k = 0;; k++) {
        const int st = k % G::kStages;
        // odd steps sweep the tiles backwards: what the last step wrote last is
        // read first, out of L2 where it still lies (128^3 FP32 with a chain
        // 63.2 -> 61.6 us a step; larger boxes lose nothing)
        const int64_t t = back && next < p.total_tiles ? p.total_tiles - 1 - next : next;
        Tile& th = hd->t[k % (2 * G::kStages)];
        // the stage's previous tile must be released by all consumer warps; if
        // that does not happen within the limit the consumers have left
        if (k >= G::kStages) {
            bool ok = true;
            if (lane == 0) ok = mbar_wait_bounded(&hd->empty[st], (uint32_t)(((k / G::kStages) - 1) & 1), p.wait_ns);
            if (!__shfl_sync(0xffffffffu, ok, 0)) return;
        }
        if (t >= p.total_tiles) {
            if (lane == 0) {
                th.box = -1;
                mbar_arrive(&hd->full[st]);  // completes the phase with no bytes: end of work
            }
            // no tile left for this block: the kernel after this one (a
            // programmatic dependent) may be scheduled once every block has
            // got here; it waits on the device for this grid to complete
            asm volatile("griddepcontrol.launch_dependents;");
            return;
        }
        long long claimed = 0;
        if (left == 1 && lane == 0)
            claimed = dealt + (long long)atomicAdd(ctr, (unsigned long long)run);  // overlaps this tile's copies
        if (t < tile_lo || t >= tile_hi) {  // another box: its record and what the collision and the boundary need at this step
            const int b = locate_box_warp(p, t, lane);
            tile_lo = only ? 0 : p.tile_prefix[b];
            tile_hi = only ? p.total_tiles : p.tile_prefix[b + 1];
            if (lane < (int)(sizeof(BoxDev) / 8))
                reinterpret_cast<uint64_t*>(&th.bd)[lane] =
                    only ? only_word : reinterpret_cast<const uint64_t*>(p.boxes + b)[lane];
            const int frozen = p.status[b] != 0;
            __syncwarp();
            if (lane == 0) {
                const TimeWeights<R> tw = time_weights<R>(n, th.bd.K, th.bd.time_interp, p.ring_slots);
                th.mlp_s = th.bd.mlp_row >= 0 ? mlp_substep(n, th.bd.K) : 0;
                if (KIND > 0 && th.bd.frame) {  // the header carries the body acceleration of step n (frame
                                                // boxes carry a body force, so they run a general kernel)
                    double a[3];
                    frame_accel_at(th.bd, p.faccel, p.ring_slots, n, a);
                    for (int c = 0; c < 3; c++) th.bd.accel[c] = a[c];
                }
                th.step = n;
                th.box = b;
                th.frozen = frozen;
                for (int a = 0; a < 4; a++) {
                    th.slot[a] = tw.slot[a];
                    th.c[a] = tw.c[a];
                }
                th.om = A(1) / (A)th.bd.tau;
                th.om1 = A(1) - th.om;
                th.srcfac = A(1) - A(0.5) * th.om;
                th.drho_b = (A)th.bd.rho_b - A(1);
                for (int c = 0; c < 3; c++) th.acc[c] = (A)th.bd.accel[c];
            }
            __syncwarp();
            Ei = th.bd.E;
            fe = Ei * Ei;
            n3 = th.bd.n3;
            div_magic = th.bd.div_magic;
            shift = cy * Ei + cz * fe + H;
            row_src = reinterpret_cast<const E*>(p.A) + th.bd.f_off + (int64_t)(lane < kQ ? lane : 0) * n3;
            ms = th.mlp_s;
            mlp = th.bd.mlp_row >= 0 && ms > 0;
            if constexpr (G::kEdges) {
                edge_src = edge_runs<G::kEdgeBytes>(p, th, T, lane, edge_last);
                __syncwarp();
                edge_bytes = edge_src ? th.edge_stride * 4 : 0;
            }
            __syncwarp();
#pragma unroll
            for (int q = 0; q < kMine; q++)
                if (lane + 32 * q < kWords) hw[q] = reinterpret_cast<const uint64_t*>(&th)[lane + 32 * q];
            __syncwarp();
        }
        const int64_t s0 = (t - tile_lo) * T;
        int edge_first = 0;
        if constexpr (G::kEdges) edge_first = min(div_e(s0, div_magic) & ~3, edge_last);
        // the header, with this tile's own words
#pragma unroll
        for (int q = 0; q < kMine; q++) {
            const int w = lane + 32 * q;
            if (w < kWords) {
                uint64_t v = hw[q];
                if (w == (int)(offsetof(Tile, s0) / 8)) v = (uint64_t)s0;
                if (w == (int)(offsetof(Tile, edge_row) / 8)) {
                    const uint64_t r = (uint32_t)edge_first;
                    v = offsetof(Tile, edge_row) % 8 ? (v & 0xffffffffull) | (r << 32) : (v & ~0xffffffffull) | r;
                }
                reinterpret_cast<uint64_t*>(&th)[w] = v;
            }
        }
        // row `lane`: source range clamped to the box's arrays
        unsigned char* stage = smem + kStagedHeaderBytes + st * (G::kStageBytes + G::kEdgeBytes);
        const int64_t start = s0 - shift;
        const int64_t lo = start > 0 ? start : 0;
        const int64_t hi = start + W < n3 ? start + W : n3;
        const bool mine = lane < kQ && hi > lo;
        const uint32_t bytes = mine ? (uint32_t)((hi - lo) * sizeof(E)) : 0u;
        if (lane < kQ) {
            const int a = mine ? (int)(lo - start) : W;  // first copied element
            const int e = mine ? (int)(hi - start) : W;  // end of the copied elements
            if (a > 0 || e < W) {
                uint4* row = reinterpret_cast<uint4*>(stage + lane * G::kRowStride);
                constexpr int per16 = 16 / (int)sizeof(E);
                for (int x = 0; x < a; x += per16) row[x / per16] = make_uint4(0, 0, 0, 0);
                for (int x = e; x < W; x += per16) row[x / per16] = make_uint4(0, 0, 0, 0);
            }
        }
        const uint32_t total = __reduce_add_sync(0xffffffffu, bytes + (uint32_t)edge_bytes);
        __syncwarp();  // header and zeroed parts written before the stage is armed
        if (t == p.withhold_tile) {
            // test only: this stage is never armed and no copy is issued, so
            // its full barrier never completes and the consumers' bounded wait
            // runs out (the header above is in place for them to name the box)
            __threadfence_block();
        } else {
            if (lane == 0) mbar_arrive_expect_tx(&hd->full[st], total);
            __syncwarp();
            if (mine) {
                fence_proxy_async_smem();
                unsigned char* dst = stage + lane * G::kRowStride + (lo - start) * sizeof(E);
                if (p.hint_loads) bulk_load_hint(dst, row_src + lo, bytes, &hd->full[st], pol);
                else bulk_load(dst, row_src + lo, bytes, &hd->full[st]);
            }
            if (edge_bytes)
                bulk_load(stage + G::kStageBytes + lane * edge_bytes, edge_src + edge_first, (uint32_t)edge_bytes, &hd->full[st]);
            // upsampler boxes: the residuals the tile's boundary sites will add
            // come from an output far larger than L2; prefetch them into L2 while
            // the copies are in flight, so that the consumers' loads hit there
            if (mlp) prefetch_mlp_residuals(p, th.bd, ms, s0, T, lane, th.edge_stride != 0);
        }
        if (--left > 0) {
            next++;
        } else {
            next = __shfl_sync(0xffffffffu, claimed, 0);
            left = run;
        }
    }
}

// KIND 0: every box of the launch is plain (velocity faces, no body force);
// 1: some box is periodic or carries a body force; 2: some box also takes the
// fluctuating collision.  Each kind compiles only the tile bodies it can meet.
template <int ST, int SPT, int KIND>
__global__ void __launch_bounds__(kStagedThreads, 1) k_stream_collide_staged(SCParams p)
{
    using G = Staged<ST, SPT>;
    extern __shared__ __align__(128) unsigned char smem[];
    StagedHeader<ST>* hd = reinterpret_cast<StagedHeader<ST>*>(smem);
    if (threadIdx.x == 0) {
        for (int st = 0; st < G::kStages; st++) {
            mbar_init(&hd->full[st], 1);
            mbar_init(&hd->empty[st], kStagedConsumerWarps);
        }
        fence_mbar_init();
    }
    __syncthreads();
    if (threadIdx.x >= kStagedConsumers) {
        staged_produce<ST, SPT, KIND>(p, smem, hd);  // the whole last warp
        // Without chains no forced re-collision follows: the last block to run
        // out of tiles ends the step (only producers claim tiles or read the
        // step, and all are done then; a producer that gave up counts as well).
        if (p.ends_step && (threadIdx.x & 31) == 0) {
            unsigned long long* ctr = reinterpret_cast<unsigned long long*>(p.tile_counter);
            __threadfence();
            if (atomicAdd(ctr + 1, 1ull) == gridDim.x - 1) {
                ctr[0] = 0;
                ctr[1] = 0;
                *const_cast<int64_t*>(p.step) += 1;
            }
        }
        return;
    }
    // the consumers' own reads of global memory also come after the kernel before
    asm volatile("griddepcontrol.wait;" ::: "memory");
    staged_consume<ST, SPT, KIND>(p, smem, hd);
}

}  // namespace lbt
