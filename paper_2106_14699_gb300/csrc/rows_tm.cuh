// Inverse row transform + fused entropy epilogue, FP32, one warp per pair
// transform (L = Q/2 = 256, 512 or 1024 points; two or three warps for 2048, 768 and 1536), with
//   * the B-marginal accumulators C_B^b(p) held in Tensor Memory (TMEM,
//     tcgen05.ld / tcgen05.st), one 32-bit column per (b, position) of the
//     owning thread, and
//   * each team's next Y row gathered into shared memory by a TMA tensor copy
//     (cp.async.bulk.tensor + mbarrier) while the current round computes.
// Same arithmetic and outputs as k_pair_rows (kernels.cuh), except the debug
// count maps: a call that asks for them runs k_pair_rows.
#pragma once
#include <cuda.h>
#include "kernels.cuh"

namespace cmif {

// ---- mbarrier / TMA bulk copy ------------------------------------------------
__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_fence_init() {
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
__device__ __forceinline__ void fence_proxy_async_smem() {
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}
// Row `row` of pair `pair` (layout of Y): the 32-byte pieces (row % 4) of the row group's
// 128-byte lines, one per chunk.  Tensor: 32 floats x L/4 chunks x row groups x pairs, boxes of
// 8 x (at most 256 chunks) x 1 x 1; x = 8 (row % 4) is a multiple of 4 floats (16 bytes).
__host__ __device__ constexpr int row_box(int L) { return L / 4 <= 256 ? L / 4 : L / 8; }
template <int L>
__device__ __forceinline__ void tma_row_g2s(uint32_t dst, const CUtensorMap* map, int row, int pair, uint32_t bar) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"((uint32_t)L * 8u) : "memory");
#pragma unroll
    for (int c = 0; c < L / 4; c += row_box(L))
        asm volatile("cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5, %6}], [%2];"
                     ::"r"(dst + 32u * c), "l"(map), "r"(bar), "r"(8 * (row & 3)), "r"(c), "r"(row >> 2), "r"(pair) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t phase) {
    uint32_t done;
    asm volatile("{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
                 : "=r"(done) : "r"(bar), "r"(phase) : "memory");
    return done != 0;
}
// Bounded wait: gives up after `polls` polls (by default 2^24, far beyond any
// copy's latency) and returns false, so that a lost copy can never hang the GPU.
constexpr int kDefaultWaitPolls = 1 << 24;
__device__ __forceinline__ bool mbar_wait_bounded(uint32_t bar, uint32_t phase, int polls = kDefaultWaitPolls) {
    for (int it = 0; it < polls; ++it)
        if (mbar_try_wait(bar, phase)) return true;
    return false;
}

// ---- Tensor Memory ------------------------------------------------------------
__device__ __forceinline__ void tmem_alloc(uint32_t dst_smem, uint32_t ncols) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(dst_smem), "r"(ncols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}
__device__ __forceinline__ void tmem_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tmem_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tmem_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void tmem_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

template <int N>
__device__ __forceinline__ void tmem_ld(uint32_t taddr, uint32_t (&r)[N]);
template <int N>
__device__ __forceinline__ void tmem_st(uint32_t taddr, const uint32_t (&r)[N]);

template <>
__device__ __forceinline__ void tmem_ld<1>(uint32_t t, uint32_t (&r)[1]) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x1.b32 {%0}, [%1];" : "=r"(r[0]) : "r"(t) : "memory");
}
template <>
__device__ __forceinline__ void tmem_st<1>(uint32_t t, const uint32_t (&r)[1]) {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x1.b32 [%0], {%1};" ::"r"(t), "r"(r[0]) : "memory");
}
template <>
__device__ __forceinline__ void tmem_ld<2>(uint32_t t, uint32_t (&r)[2]) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x2.b32 {%0, %1}, [%2];" : "=r"(r[0]), "=r"(r[1]) : "r"(t) : "memory");
}
template <>
__device__ __forceinline__ void tmem_st<2>(uint32_t t, const uint32_t (&r)[2]) {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x2.b32 [%0], {%1, %2};" ::"r"(t), "r"(r[0]), "r"(r[1]) : "memory");
}
#define CMIF_R16(o) "=r"(r[o]), "=r"(r[o + 1]), "=r"(r[o + 2]), "=r"(r[o + 3]), "=r"(r[o + 4]), "=r"(r[o + 5]), \
    "=r"(r[o + 6]), "=r"(r[o + 7]), "=r"(r[o + 8]), "=r"(r[o + 9]), "=r"(r[o + 10]), "=r"(r[o + 11]),           \
    "=r"(r[o + 12]), "=r"(r[o + 13]), "=r"(r[o + 14]), "=r"(r[o + 15])
#define CMIF_W16(o) "r"(r[o]), "r"(r[o + 1]), "r"(r[o + 2]), "r"(r[o + 3]), "r"(r[o + 4]), "r"(r[o + 5]), \
    "r"(r[o + 6]), "r"(r[o + 7]), "r"(r[o + 8]), "r"(r[o + 9]), "r"(r[o + 10]), "r"(r[o + 11]),           \
    "r"(r[o + 12]), "r"(r[o + 13]), "r"(r[o + 14]), "r"(r[o + 15])
template <>
__device__ __forceinline__ void tmem_ld<4>(uint32_t t, uint32_t (&r)[4]) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(t) : "memory");
}
template <>
__device__ __forceinline__ void tmem_st<4>(uint32_t t, const uint32_t (&r)[4]) {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x4.b32 [%0], {%1, %2, %3, %4};"
                 ::"r"(t), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]) : "memory");
}
#define CMIF_R8(o) "=r"(r[o]), "=r"(r[o + 1]), "=r"(r[o + 2]), "=r"(r[o + 3]), "=r"(r[o + 4]), "=r"(r[o + 5]), \
    "=r"(r[o + 6]), "=r"(r[o + 7])
#define CMIF_W8(o) "r"(r[o]), "r"(r[o + 1]), "r"(r[o + 2]), "r"(r[o + 3]), "r"(r[o + 4]), "r"(r[o + 5]), \
    "r"(r[o + 6]), "r"(r[o + 7])
template <>
__device__ __forceinline__ void tmem_ld<8>(uint32_t t, uint32_t (&r)[8]) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : CMIF_R8(0) : "r"(t) : "memory");
}
template <>
__device__ __forceinline__ void tmem_st<8>(uint32_t t, const uint32_t (&r)[8]) {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};"
                 ::"r"(t), CMIF_W8(0) : "memory");
}
#undef CMIF_R8
#undef CMIF_W8
template <>
__device__ __forceinline__ void tmem_ld<16>(uint32_t t, uint32_t (&r)[16]) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, "
                 "%14, %15}, [%16];"
                 : CMIF_R16(0) : "r"(t) : "memory");
}
template <>
__device__ __forceinline__ void tmem_st<16>(uint32_t t, const uint32_t (&r)[16]) {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, "
                 "%13, %14, %15, %16};"
                 ::"r"(t), CMIF_W16(0) : "memory");
}
template <>
__device__ __forceinline__ void tmem_ld<32>(uint32_t t, uint32_t (&r)[32]) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, "
                 "%14, %15, %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
                 : CMIF_R16(0), CMIF_R16(16) : "r"(t) : "memory");
}
template <>
__device__ __forceinline__ void tmem_st<32>(uint32_t t, const uint32_t (&r)[32]) {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, "
                 "%13, %14, %15, %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31, %32};"
                 ::"r"(t), CMIF_W16(0), CMIF_W16(16) : "memory");
}
#undef CMIF_R16
#undef CMIF_W16

// ---------------------------------------------------------------------------
// The warp's transform of L = 32 PTS points (PTS = 8, 16, 32 per lane), four-step:
// lane j holds x[j + 32 i], i < PTS; a PTS-point DFT over i gives rows k1 < PTS; twiddle
// w_L^{j k1}; a transpose through the warp's buffer (PTS rows of 32 floats, real plane then
// imaginary plane, blocks of 4 floats XOR-permuted by the row: conflict-free 16-byte row
// reads); then a 32-point DFT along each row by RS = 32 / PTS lanes, lane k1 + PTS r taking
// the outputs k2 = RS q + r: each loads the whole row, forms its radix-RS combination
// y_r[n] = w_32^{nr} sum_s i^{sr..} x[n + PTS s] and a second PTS-point DFT.  So output q of lane l
// is X[l + 32 q] for every PTS, and no step but the transpose leaves the registers.  All
// DFTs are packed (fft_pk.cuh): re[m] = values 2m, 2m + 1 on entry, q and q + PTS/2 on exit.
// tw1[k 32 + j]: w_L^{j k}, w_L^{j (k + PTS/2)}; tw2[r PTS/2 + m]: w_32^{2m r}, w_32^{(2m+1) r},
// both as (cos, cos', sin, sin') with the forward sign.
__device__ __forceinline__ void mul_conj2(float2& re, float2& im, float4 w) {
    const float2 c = make_float2(w.x, w.y), s = make_float2(w.z, w.w), a = re, b = im;
    re = __ffma2_rn(b, s, __fmul2_rn(a, c));
    im = __fmul2_rn(b, c);
    im = make_float2(fmaf(-a.x, s.x, im.x), fmaf(-a.y, s.y, im.y));
}
template <int PTS>
__device__ __forceinline__ void warp_fft_inv(float2 (&re)[PTS / 2], float2 (&im)[PTS / 2], int lane, float* sf,
                                             const float4* tw1, const float4* tw2) {
    constexpr int H = PTS / 2, RS = 32 / PTS;
    dft_pk<PTS, +1>(re, im);
#pragma unroll
    for (int k = 0; k < H; ++k) mul_conj2(re[k], im[k], tw1[k * 32 + lane]);
    float* si = sf + PTS * 32;
    __syncwarp();
#pragma unroll
    for (int x = 0; x < 8; ++x) {  // rows x, x + 8, .. share a block permutation: one address
        char* const p = reinterpret_cast<char*>(sf) + ((lane << 2) ^ (x << 4));
#pragma unroll
        for (int row = x; row < PTS; row += 8) {
            *reinterpret_cast<float*>(p + row * 128) = row < H ? re[row].x : re[row - H].y;
            *reinterpret_cast<float*>(p + row * 128 + PTS * 128) = row < H ? im[row].x : im[row - H].y;
        }
    }
    __syncwarp();
    const int k1 = lane & (PTS - 1), r = lane / PTS;
    auto block = [&](const float* pl, int b) {
        return *reinterpret_cast<const float4*>(pl + k1 * 32 + (((b ^ k1) & 7) << 2));
    };
    auto lo = [](float4 q) { return make_float2(q.x, q.y); };
    auto hi = [](float4 q) { return make_float2(q.z, q.w); };
    if constexpr (RS == 1) {
#pragma unroll
        for (int b = 0; b < 8; ++b) {
            const float4 p = block(sf, b), q = block(si, b);
            re[2 * b] = lo(p); re[2 * b + 1] = hi(p);
            im[2 * b] = lo(q); im[2 * b + 1] = hi(q);
        }
    } else if constexpr (RS == 2) {
        const float sg = r ? -1.f : 1.f;
#pragma unroll
        for (int b = 0; b < 4; ++b) {
            const float4 p0 = block(sf, b), p1 = block(sf, b + 4), q0 = block(si, b), q1 = block(si, b + 4);
            re[2 * b] = fmak(lo(p1), sg, lo(p0)); re[2 * b + 1] = fmak(hi(p1), sg, hi(p0));
            im[2 * b] = fmak(lo(q1), sg, lo(q0)); im[2 * b + 1] = fmak(hi(q1), sg, hi(q0));
        }
    } else {
        static_assert(RS == 4, "8, 16 or 32 points per lane");
        // (x0 + (-1)^r x2) + i^r (x1 + (-1)^r x3)
        const float sg = (r & 1) ? -1.f : 1.f, cr = r == 0 ? 1.f : r == 2 ? -1.f : 0.f, ci = r == 1 ? 1.f : r == 3 ? -1.f : 0.f;
        auto join = [&](float2 x0, float2 x1, float2 x2, float2 x3, float2 y0, float2 y1, float2 y2, float2 y3,
                        float2& zr, float2& zi) {
            const float2 ar = fmak(x2, sg, x0), br = fmak(x3, sg, x1), ai = fmak(y2, sg, y0), bi = fmak(y3, sg, y1);
            zr = fmak(bi, -ci, fmak(br, cr, ar));
            zi = fmak(br, ci, fmak(bi, cr, ai));
        };
#pragma unroll
        for (int b = 0; b < 2; ++b) {
            const float4 p0 = block(sf, b), p1 = block(sf, b + 2), p2 = block(sf, b + 4), p3 = block(sf, b + 6);
            const float4 q0 = block(si, b), q1 = block(si, b + 2), q2 = block(si, b + 4), q3 = block(si, b + 6);
            join(lo(p0), lo(p1), lo(p2), lo(p3), lo(q0), lo(q1), lo(q2), lo(q3), re[2 * b], im[2 * b]);
            join(hi(p0), hi(p1), hi(p2), hi(p3), hi(q0), hi(q1), hi(q2), hi(q3), re[2 * b + 1], im[2 * b + 1]);
        }
    }
    if constexpr (RS > 1) {
#pragma unroll
        for (int m = 0; m < H; ++m) mul_conj2(re[m], im[m], tw2[r * H + m]);
    }
    __syncwarp();  // the buffer's reads are done
    dft_pk<PTS, +1>(re, im);
}

// L = G LS: a team of G warps.  G = 2, 3 (Q = 4096, 1536, 3072): radix-G decimation in frequency as
// the values are loaded: warp r forms y_r[m] = w_L^{mr} sum_s w_G^{sr} x[m + s LS] and transforms
// its LS points; X[G k + r] = Y_r[k].  Against the generic kernel (which keeps a whole row's
// counts and marginals in shared memory: one or two blocks of idle FMA pipes), rows of 300-row
// maps, four angles, ms: Q = 3072, 8 x 8 labels 1.64 -> 1.03, 16 x 16 6.42 -> 3.84 (2.9 -> 4.9e11
// counts/s); Q = 4096 2.74 -> 1.15, 13.6 -> 4.24; Q = 1536, 36 x 36 15.2 -> 12.8.  Every warp of a
// team reads the whole row (G shared-memory reads of each value), which costs most at G = 3.
// NT teams per block, BLOCKS blocks per SM.  Narrow rows hold few values per lane, so
// more warps fit, and several small blocks, each with its own barriers, run one's transforms
// (FMA pipe) beside another's entropy terms (ALU, MUFU).  Measured at K = 16 (1e11 counts/s):
// Q = 512: 16 warps in one block 5.0, 2 blocks of 8 5.8, 4 of 8 6.2; Q = 1024: one of 16 6.5,
// 2 of 8 7.0, 3 of 8 (spills) 4.8; Q = 2048: one of 16 7.0, 2 of 8 7.1 (1024 x 1024; few rows:
// rows_tm_teams).  NT = 16 also where two blocks' marginals do not fit in Tensor Memory.
template <int Q, int NT_>
struct RowTmCfg {
    static constexpr int L = Q / 2, G = Q % 3 == 0 ? 3 : Q == 4096 ? 2 : 1, LS = L / G;
    static constexpr int PTS = LS / 32, H = PTS / 2, RS = 32 / PTS;
    static constexpr int NT = NT_, WARPS = NT * G, THREADS = WARPS * 32;
    static constexpr int BLOCKS = Q == 1536 ? 2 : G > 1 || NT == 16 ? 1 : Q == 512 ? 4 : 2;
    // one pass holds the whole row: fewer barriers and TMEM round trips per round; at 2048 and
    // 4096 the counts of a round go to their owners in two passes
    static constexpr int HALVES = Q == 2048 || Q == 4096 ? 2 : 1;
    static constexpr int QH = Q / HALVES;        // positions per pass
    static constexpr int UH = QH / THREADS;      // positions per thread per pass: adjacent floats of the hand-over
    static constexpr int U = HALVES * UH;
    static constexpr int REGION = QH * 4;        // one pass of a pair's rounded counts: G parts, one per warp
    static constexpr int STAGE_BYTES = L * 8;    // one Y row, then the warps' transpose planes
    static constexpr size_t OFF_STAGE = (size_t)NT * REGION;
    static constexpr size_t OFF_BAR = OFF_STAGE + (size_t)NT * STAGE_BYTES;
    static constexpr size_t OFF_HOLD = OFF_BAR + 16 * 8;
    static constexpr size_t OFF_TW1 = OFF_HOLD + 16;                       // twiddles, as float4
    static constexpr size_t OFF_TW2 = OFF_TW1 + (size_t)H * 32 * 16;
    static constexpr size_t OFF_TW3 = OFF_TW2 + (RS > 1 ? (size_t)RS * H * 16 : 0);
    static constexpr size_t SMEM = OFF_TW3 + (size_t)(G - 1) * H * 32 * 16;
    // B-marginals per TMEM round trip: as many as the registers hold beside the second pass's counts
    static constexpr int NMED = UH == 8 || (UH == 4 && HALVES == 2) ? 4 : 8, NBIG = UH <= 2 ? 16 : NMED;
    static_assert(UH == 1 || UH == 2 || UH == 4 || UH == 8, "positions per thread and pass");
    static_assert((size_t)NT * REGION >= (size_t)Q * 12, "the hand-over region holds a row of MI and N");
    static_assert(PTS * 32 * 8 * G <= STAGE_BYTES, "a warp's planes fit its part of the staged row");
    // Position (0 .. Q) of float f of pass hf in a pair's hand-over region: part r (warp); its slot
    // f / 2 of lane l = slot % 32 holds values q and q + H of the lane, real or imaginary part
    static __device__ __forceinline__ int position(int hf, int f) {
        constexpr int PART = QH / G;
        const int r = G == 1 ? 0 : f / PART, fr = f - r * PART;
        const int slot = fr >> 1, l = slot & 31, qc = slot >> 5;
        const int q = hf * (H / HALVES) + (qc >> 1) + (fr & 1) * H;
        return 2 * (G * (l + 32 * q) + r) + (qc & 1);
    }
};

// A barrier over the G warps of one team (G = 1: the warp).
template <int G>
__device__ __forceinline__ void team_sync(int team) {
    if constexpr (G == 1) __syncwarp();
    else asm volatile("bar.sync %0, %1;" ::"r"(1 + team), "r"(G * 32) : "memory");
}

// The order of the pairs: label a outside, b inside, or, for the wide rows of several-warp teams
// with fewer labels a, the other way round (more inputs fit in Tensor Memory).  Not for the
// one-warp teams, whose kernel is at the register limit: Q = 2048, 24 x 24 labels 3.79 ms
// without, 3.91 ms with the choice.
__host__ __device__ constexpr bool tm_swapped(int Q, int KA, int KB) { return (Q % 3 == 0 || Q == 4096) && KA < KB; }
// TMEM columns a block needs: KI marginals (the inner labels) x U = Q / (32 WARPS) positions per
// thread, WARPS / 4 warps per lane quadrant.
__host__ __device__ constexpr int tm_cols_needed(int KI, int Q) { return KI * (Q / 128); }
__host__ __device__ constexpr int tm_alloc_cols(int need) {
    return need <= 32 ? 32 : need <= 64 ? 64 : need <= 128 ? 128 : need <= 256 ? 256 : 512;
}

// MODE 0 is the plain FP32 kernel (one map); MODE 1 takes several units per
// launch (rotation angles); MODE 2 adds to that the per-pair precision of
// CMIF_AUTO (conditional re-run, exact counts of listed pairs, per-pair
// residuals) and the diagnostics of the bounded waits (poll limit, withheld
// copy).  They are separate instantiations because the plain kernel sits at
// the register limit.
template <int Q, bool NMI, int MODE, int NTEAMS>
__global__ void __launch_bounds__(RowTmCfg<Q, NTEAMS>::THREADS, RowTmCfg<Q, NTEAMS>::BLOCKS)
k_pair_rows_tm(const __grid_constant__ CUtensorMap ymap, Geom g, Tw<float> tw, double* __restrict__ mi_map,
               int32_t* __restrict__ n_map, DevStatus* __restrict__ st,
               int tm_cols, int wait_polls, int withhold_row, int conditional, const int32_t* __restrict__ ov,
               const int* __restrict__ ov_slot, unsigned* __restrict__ pair_res) {
    // wait_polls: poll limit of the bounded waits.  withhold_row >= 0 (diagnostics
    // only): the bulk copy of that output row's first pair is never issued, so the
    // wait for it runs out and the kernel takes its timeout path.  conditional: run
    // only when the status word asks for the re-run.  ov, ov_slot, pair_res: the
    // exact counts of second-precision pairs and the per-pair residuals, as in
    // k_pair_rows.
    using C = RowTmCfg<Q, NTEAMS>;
    constexpr bool EXT = MODE == 2, MULTI = MODE >= 1;
    if (EXT && conditional && !(st->flags & STATUS_ESCALATE)) return;  // uniform, before any set-up
    if (!EXT) {
        wait_polls = kDefaultWaitPolls;
        withhold_row = -1;
    }
    constexpr int L = C::L, NT = C::NT, U = C::U, UH = C::UH, HALVES = C::HALVES, PTS = C::PTS, H = C::H, G = C::G;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, team = warp / G, wr = warp % G;  // warp wr of the team
    float2* region = reinterpret_cast<float2*>(smem_raw + (size_t)team * C::REGION + (size_t)wr * (C::REGION / G));
    float* stage = reinterpret_cast<float*>(smem_raw + C::OFF_STAGE + (size_t)team * C::STAGE_BYTES);
    const uint32_t stage_s = smem_u32(stage);
    const uint32_t bar = smem_u32(smem_raw + C::OFF_BAR + team * 8);
    uint32_t* hold = reinterpret_cast<uint32_t*>(smem_raw + C::OFF_HOLD);

    // pairs in runs of one outer label: its marginal in registers, the KI inner labels' in TMEM
    const int npairs = g.KA * g.KB, Rout = g.R, Cout = g.C;
    const bool swapped = tm_swapped(Q, g.KA, g.KB);
    const int KI = swapped ? g.KA : g.KB;
    auto pair_id = [&](int t) {  // pair t in this order -> a * K_B + b
        if (!swapped) return t;
        const int o = t / KI;
        return (t - o * KI) * g.KB + o;
    };
    float4* tw1 = reinterpret_cast<float4*>(smem_raw + C::OFF_TW1);
    float4* tw2 = reinterpret_cast<float4*>(smem_raw + C::OFF_TW2);
    for (int i = tid; i < H * 32; i += C::THREADS) {
        const int k = i >> 5, j = i & 31;
        const cpx<float> a = tw_of<C::LS>(tw)[j * k], b = tw_of<C::LS>(tw)[j * (k + H)];
        tw1[i] = make_float4(a.x, b.x, a.y, b.y);
    }
    if (C::RS > 1) {
        for (int i = tid; i < C::RS * H; i += C::THREADS) {
            const int r = i / H, m = i % H;
            const cpx<float> a = tw_of<32>(tw)[2 * m * r], b = tw_of<32>(tw)[(2 * m + 1) * r];
            tw2[i] = make_float4(a.x, b.x, a.y, b.y);
        }
    }

    float4* tw3 = reinterpret_cast<float4*>(smem_raw + C::OFF_TW3);  // w_L^{mr} of lane j's pairs, r >= 1
    if (G > 1) {
        for (int i = tid; i < (G - 1) * H * 32; i += C::THREADS) {
            const int r = i / (H * 32) + 1, m = (i >> 5) % H, n = (i & 31) + 64 * m;
            const cpx<float> a = tw_of<L>(tw)[n * r], b = tw_of<L>(tw)[(n + 32) * r];
            tw3[i] = make_float4(a.x, b.x, a.y, b.y);
        }
    }
    if (lane == 0 && wr == 0) mbar_init(bar, 1);
    if (warp == 0) tmem_alloc(smem_u32(hold), (uint32_t)tm_cols);
    mbar_fence_init();
    tmem_fence_before();
    __syncthreads();
    tmem_fence_after();
    const uint32_t tmem = *hold;
    // this warp's TMEM slice: lanes of quadrant (warp % 4), columns of block (warp / 4)
    const uint32_t tbase = tmem + ((uint32_t)(32 * (warp & 3)) << 16) + (uint32_t)((warp >> 2) * KI * U);

    // work items of this team: (row, base) in order; prefetch the first active one
    uint32_t phase = 0;
    bool pending = false;  // a copy issued for this team and not yet waited for
    // work: tasks blockIdx.x + k * gridDim.x of the window's rows; several units (maps, R2
    // rows apart) form one run of tasks, so that the last round of blocks is short once
    // and not once per unit.  One unit is the whole map: a volume's R = Dz R2 rows.
    const int nr = g.r1 - g.r0, unit_rows = g.units > 1 ? g.R2 : Rout;
    auto advance = [&](int& rr, int& base) {  // task offset rr within its unit, the unit's first row
        while (rr >= g.r1) {
            rr -= nr;
            base += unit_rows;
        }
    };
    auto issue = [&](int row_i, int pair_i) {
        if (EXT && row_i == withhold_row && pair_i == 0) return;  // diagnostics: leave this wait without its copy
        if (lane == 0 && wr == 0) {
            fence_proxy_async_smem();
            tma_row_g2s<L>(stage_s, &ymap, row_i, pair_id(pair_i), bar);
        }
        pending = true;
    };
    int rr = g.r0 + (int)blockIdx.x, rbase = 0;  // row of the first unit's window; unit * unit_rows (multi-unit kernels)
    if (MULTI) advance(rr, rbase);
    if (MULTI ? rbase < g.R : rr < g.r1) {
        if (team < npairs) issue(rbase + rr, team);
    }

    float res_max = 0.f;
    int row_max_n = 0;
    bool aborted = false;
    while ((MULTI ? rbase < g.R : rr < g.r1) && !aborted) {
        const int row = MULTI ? rbase + rr : rr;
        EntAcc<NMI> S[U];
        float CA[U];
#pragma unroll
        for (int u = 0; u < U; ++u) { S[u].zero(); CA[u] = 0.f; }
        {   // zero this thread's B-marginal columns
            uint32_t z[16];
#pragma unroll
            for (int i = 0; i < 16; ++i) z[i] = 0u;
            for (int c0 = 0; c0 < KI * U; c0 += 16) {
                if (c0 + 16 <= KI * U) tmem_st<16>(tbase + c0, z);
                else for (int c = c0; c < KI * U; ++c) { uint32_t z1[1] = {0u}; tmem_st<1>(tbase + c, z1); }
            }
            tmem_wait_st();
        }
        int cur_a[2] = {0, 0};
        for (int base = 0; base < npairs; base += NT) {
            const int pair = base + team;
            const bool act = pair < npairs;
            // A team without a pair in this round leaves its buffer alone (the copy of its
            // next row's pair may be in flight into it); its counts are never read.
            float2 re[H], im[H];
            int timeout = 0;
            if (act) {
                if (mbar_wait_bounded(bar, phase, wait_polls)) {
                    phase ^= 1u;
                    pending = false;
                } else {
                    atomicOr(&st->flags, STATUS_TIMEOUT);
                    timeout = 1;
                }
                // the lane's inputs z[lane + 32 i] in pairs (layout of Y, kernels.cuh): the
                // direct halves of chunks 32 m + lane, then the mirrored halves of lane -lane
                const float4* sg4 = reinterpret_cast<const float4*>(stage);
                const int jj = (32 - lane) & 31;
                const float4* dsrc = sg4 + 2 * lane + ((lane >> 2) & 1);
                const float4* msrc = sg4 + 2 * jj + (1 ^ ((jj >> 2) & 1));
                constexpr int HP = G * H / 2;  // direct pairs of the row
                auto raw = [&](int u) { return u < HP ? dsrc[64 * u] : msrc[64 * (2 * HP - 1 - u)]; };
                // Column 0's mirrors come in the other order and one pair off (its own mirror is
                // L / 2): lane 0's even inputs are the previous pair's second values.
                if constexpr (G == 1) {
#pragma unroll
                    for (int m = 0; m < H; ++m) {
                        const float4 x = raw(m);
                        re[m] = make_float2(x.x, x.y);
                        im[m] = make_float2(x.z, x.w);
                    }
                    float pr = re[H - 1].y, pi = im[H - 1].y;
#pragma unroll
                    for (int m = H / 2; m < H; ++m) {
                        const float2 tr = re[m], ti = im[m];
                        re[m].x = lane == 0 ? pr : tr.x;
                        im[m].x = lane == 0 ? pi : ti.x;
                        re[m].y = lane == 0 ? tr.x : tr.y;
                        im[m].y = lane == 0 ? ti.x : ti.y;
                        pr = tr.y;
                        pi = ti.y;
                    }
                } else {
                    float2 prev[G];  // the raw pair before the next one of the row's part s
                    auto input = [&](int s, int m) {
                        const int u = s * H + m;
                        float4 x = raw(u);
                        if (u >= HP) {
                            if (u == HP) {
                                const float4 w = raw(2 * HP - 1);
                                prev[s] = make_float2(w.y, w.w);
                            } else if (m == 0) {
                                const float4 w = raw(u - 1);
                                prev[s] = make_float2(w.y, w.w);
                            }
                            const float2 next = make_float2(x.y, x.w);
                            x = lane == 0 ? make_float4(prev[s].x, x.x, prev[s].y, x.z) : x;
                            prev[s] = next;
                        }
                        return x;
                    };
#pragma unroll
                    for (int m = 0; m < H; ++m) {
                        const float4 x0 = input(0, m);
                        if constexpr (G == 2) {
                            const float4 x1 = input(1, m);
                            const float sg = wr ? -1.f : 1.f;
                            re[m] = fmak(make_float2(x1.x, x1.y), sg, make_float2(x0.x, x0.y));
                            im[m] = fmak(make_float2(x1.z, x1.w), sg, make_float2(x0.z, x0.w));
                        } else {
                            // x0 + w_3^r x1 + w_3^{2r} x2: x0 + x1 + x2, or x0 - t/2 +- i (sqrt 3 / 2) d
                            const float4 x1 = input(1, m), x2 = input(2, m);
                            const float2 tr = addv(make_float2(x1.x, x1.y), make_float2(x2.x, x2.y));
                            const float2 ti = addv(make_float2(x1.z, x1.w), make_float2(x2.z, x2.w));
                            if (wr == 0) {
                                re[m] = addv(make_float2(x0.x, x0.y), tr);
                                im[m] = addv(make_float2(x0.z, x0.w), ti);
                            } else {
                                const float2 dr = subv(make_float2(x1.x, x1.y), make_float2(x2.x, x2.y));
                                const float2 di = subv(make_float2(x1.z, x1.w), make_float2(x2.z, x2.w));
                                const float s3 = wr == 1 ? 0.86602540378443864676f : -0.86602540378443864676f;
                                re[m] = fmak(di, -s3, fmak(tr, -0.5f, make_float2(x0.x, x0.y)));
                                im[m] = fmak(dr, s3, fmak(ti, -0.5f, make_float2(x0.z, x0.w)));
                            }
                        }
                        if (wr > 0) mul_conj2(re[m], im[m], tw3[((wr - 1) * H + m) * 32 + lane]);
                    }
                }
                if (G > 1) team_sync<G>(team);  // the team's warps have read the row: it becomes their planes
                warp_fft_inv<PTS>(re, im, lane, stage + wr * (PTS * 64), tw1, tw2);
                if (G > 1) team_sync<G>(team);  // and their planes are read
            } else {
#pragma unroll
                for (int k = 0; k < H; ++k) re[k] = im[k] = make_float2(0.f, 0.f);
            }
            // the staging buffer is free again: prefetch this team's next active item
            // (the next round of this row, else round 0 of its next row)
            if (act && !pending) {
                if constexpr (MULTI) {
                    int nb = rbase, nrr = rr, npair = pair + NT;
                    if (npair >= npairs) {
                        npair = team;
                        nrr = rr + gridDim.x;
                        advance(nrr, nb);
                    }
                    if (nb < g.R) issue(nb + nrr, npair);
                } else {
                    int nrow = row, npair = pair + NT;
                    if (npair >= npairs) { nrow = row + gridDim.x; npair = team; }
                    if (nrow < g.r1) issue(nrow, npair);
                }
            }
            float rp = 0.f;
            auto round2 = [&](float2& x) {  // nearest integers (the 1.5 * 2^23 shift) and the residual
                const float2 c = __fadd2_rn(__fadd2_rn(x, make_float2(12582912.0f, 12582912.0f)),
                                            make_float2(-12582912.0f, -12582912.0f));
                const float2 dv = subv(x, c);
                if constexpr (EXT) rp = fmaxf(rp, fmaxf(fabsf(dv.x), fabsf(dv.y)));
                else res_max = fmaxf(res_max, fmaxf(fabsf(dv.x), fabsf(dv.y)));
                x = c;
            };
#pragma unroll
            for (int k = 0; k < H; ++k) {
                round2(re[k]);
                round2(im[k]);
            }
            const int ovs = (EXT && act && ov_slot) ? ov_slot[pair_id(pair)] : -1;  // loaded after the transform: fewer live registers
            if (EXT && ovs < 0) res_max = fmaxf(res_max, rp);
            if (EXT && pair_res && act && ovs < 0) {
#pragma unroll
                for (int off = 16; off > 0; off >>= 1) rp = fmaxf(rp, __shfl_xor_sync(0xffffffffu, rp, off));
                if (lane == 0) atomic_max_float_pos(&pair_res[pair_id(pair)], rp);
            }
            const int nt = min(NT, npairs - base);
            const int a0 = base / KI, b0 = base - a0 * KI;  // outer and inner label of the round's first pair
#pragma unroll
            for (int hf = 0; hf < HALVES; ++hf) {
                if (aborted) continue;
                // every thread is done with the region's previous counts; a team whose copy
                // never came ends the block
                if (hf == 0) {
                    aborted = __syncthreads_or(timeout);
                    if (aborted) continue;
                } else {
                    __syncthreads();
                }
                constexpr int HP = H / HALVES;
                if (EXT && ovs >= 0) {  // exact counts of positions 2 z, 2 z + 1 from the second precision
                    const int32_t* ovr = ov + ((size_t)ovs * Rout + row) * Q;
#pragma unroll
                    for (int q = 0; q < HP; ++q) {
                        const int z = lane + 32 * (hf * HP + q);
                        const int2 x = *reinterpret_cast<const int2*>(ovr + 2 * (G * z + wr));
                        const int2 y = *reinterpret_cast<const int2*>(ovr + 2 * (G * (z + 32 * H) + wr));
                        region[2 * q * 32 + lane] = make_float2((float)x.x, (float)y.x);
                        region[(2 * q + 1) * 32 + lane] = make_float2((float)x.y, (float)y.y);
                    }
                } else {
#pragma unroll
                    for (int q = 0; q < HP; ++q) {
                        region[2 * q * 32 + lane] = re[hf * HP + q];
                        region[(2 * q + 1) * 32 + lane] = im[hf * HP + q];
                    }
                }
                __syncthreads();
                const uint32_t tcol = tbase + (uint32_t)(hf * KI * UH);
                // NB pairs of one label a, labels b .. b + NB - 1: their B-marginals of this pass in
                // registers, one TMEM load and store
                auto accum = [&](auto nbc, int t0, int b) {
                    constexpr int NB = decltype(nbc)::value;
                    uint32_t cbr[NB * UH];
                    tmem_ld<NB * UH>(tcol + (uint32_t)(b * UH), cbr);
                    tmem_wait_ld();
#pragma unroll
                    for (int t = 0; t < NB; ++t) {
                        const float* obt = reinterpret_cast<const float*>(smem_raw + (size_t)(t0 + t) * C::REGION);
                        if constexpr (UH == 1) {
                            const float c = obt[tid];
                            S[hf].joint(clog2c_biased(c));
                            CA[hf] += c;
                            cbr[t] = __float_as_uint(__uint_as_float(cbr[t]) + c);
                        } else {
                            float cv[UH];
                            if constexpr (UH >= 4) {
#pragma unroll
                                for (int w = 0; w < UH / 4; ++w) {
                                    const float4 q = reinterpret_cast<const float4*>(obt)[UH / 4 * tid + w];
                                    cv[4 * w] = q.x; cv[4 * w + 1] = q.y; cv[4 * w + 2] = q.z; cv[4 * w + 3] = q.w;
                                }
                            } else {
                                const float2 q = reinterpret_cast<const float2*>(obt)[tid];
                                cv[0] = q.x; cv[1] = q.y;
                            }
#pragma unroll
                            for (int w = 0; w < UH; w += 2) {
                                const float2 c = make_float2(cv[w], cv[w + 1]);
                                const int u = hf * UH + w, i = t * UH + w;
                                long long x, y;
                                clog2c_biased2(c, x, y);
                                S[u].joint(x);
                                S[u + 1].joint(y);
                                const float2 ca = __fadd2_rn(make_float2(CA[u], CA[u + 1]), c);
                                CA[u] = ca.x;
                                CA[u + 1] = ca.y;
                                const float2 m = __fadd2_rn(make_float2(__uint_as_float(cbr[i]), __uint_as_float(cbr[i + 1])), c);
                                cbr[i] = __float_as_uint(m.x);
                                cbr[i + 1] = __float_as_uint(m.y);
                            }
                        }
                    }
                    tmem_st<NB * UH>(tcol + (uint32_t)(b * UH), cbr);
                    tmem_wait_st();
                };
                int a = a0, b = b0, t = 0;
                while (t < nt) {
                    if (a != cur_a[hf]) {
#pragma unroll
                        for (int uh = 0; uh < UH; ++uh) {
                            const int u = hf * UH + uh;
                            S[u].marg(clog2c_biased(CA[u]));
                            CA[u] = 0.f;
                        }
                        cur_a[hf] = a;
                    }
                    const int seg = min(KI - b, nt - t);  // the rest of the outer label's run in this round
                    int d;
                    constexpr int NMED = C::NMED, NBIG = C::NBIG;
                    if (NBIG > NMED && seg >= NBIG) {
                        accum(std::integral_constant<int, NBIG>{}, t, b);
                        d = NBIG;
                    } else if (seg >= NMED) {
                        accum(std::integral_constant<int, NMED>{}, t, b);
                        d = NMED;
                    } else if (seg >= 2) {
                        accum(std::integral_constant<int, 2>{}, t, b);
                        d = 2;
                    } else {
                        accum(std::integral_constant<int, 1>{}, t, b);
                        d = 1;
                    }
                    t += d;
                    b += d;
                    if (b == KI) { b = 0; ++a; }
                }
            }
            if (aborted) break;
        }
        if (aborted) break;
        __syncthreads();  // the last counts are read
        // finish the row: the last outer label's marginal, the inner labels', then MI and N through the
        // hand-over region (doubles, then integers), so that the map is written in order
        double* mrow = reinterpret_cast<double*>(smem_raw);
        int* nrow_s = reinterpret_cast<int*>(smem_raw + (size_t)Q * 8);
#pragma unroll
        for (int hf = 0; hf < HALVES; ++hf) {
            float n[UH];  // N = the sum of the inner labels' marginals (exact: below 2^23)
#pragma unroll
            for (int uh = 0; uh < UH; ++uh) {
                S[hf * UH + uh].marg(clog2c_biased(CA[hf * UH + uh]));
                n[uh] = 0.f;
            }
            for (int b = 0; b < KI; ++b) {
                uint32_t cbr[UH];
                tmem_ld<UH>(tbase + (uint32_t)(hf * KI * UH + b * UH), cbr);
                tmem_wait_ld();
#pragma unroll
                for (int uh = 0; uh < UH; ++uh) {
                    const float c = __uint_as_float(cbr[uh]);
                    S[hf * UH + uh].marg(clog2c_biased(c));
                    n[uh] += c;
                }
            }
#pragma unroll
            for (int uh = 0; uh < UH; ++uh) {
                const int p = C::position(hf, UH * tid + uh), ni = (int)n[uh];
                mrow[p] = S[hf * UH + uh].finish(ni);
                nrow_s[p] = ni;
            }
        }
        __syncthreads();
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int p = tid + C::THREADS * u, cidx = circ_to_out(p, Q, g.WA, g.WB - 1);
            if (cidx < 0) continue;
            const size_t o = (size_t)row * Cout + cidx;
            const int n = nrow_s[p];
            mi_map[o] = mrow[p];
            if (n_map) n_map[o] = n;
            if (cidx >= g.c0 && cidx < g.c1) row_max_n = max(row_max_n, n);
        }
        __syncthreads();
        rr += gridDim.x;
        if (MULTI) advance(rr, rbase);
    }
    // A team may still have a copy in flight (prefetched for an item it will not run
    // after an abort): wait for it, bounded, before the block exits.
    if (pending) mbar_wait_bounded(bar, phase, wait_polls);
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        res_max = fmaxf(res_max, __shfl_xor_sync(0xffffffffu, res_max, off));
        row_max_n = max(row_max_n, __shfl_xor_sync(0xffffffffu, row_max_n, off));
    }
    if (lane == 0) {
        atomic_max_float_pos(&st->res_bits[0], res_max);
        atomicMax(&st->max_n, row_max_n);
    }
    tmem_fence_before();
    __syncthreads();
    tmem_fence_after();
    if (warp == 0) tmem_dealloc(tmem, (uint32_t)tm_cols);
}

}  // namespace cmif
