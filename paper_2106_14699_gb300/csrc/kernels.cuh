// CMIF kernels: the frequency-domain method of Sec. 3.2.
//
//   fwd_rows   : level sets L_a[X] of one label image (Sec. 3.1), two planes
//                packed per complex row FFT of length Q, unpacked into the
//                half spectra of both planes.  Also checks labels in range.
//   fwd_cols   : column FFT of length P -> 2-D half spectra F[plane][kx][ky].
//   pair_cols  : for every label pair (a, b): conj(F[L_a A]) * F[L_b B] (the
//                correlation theorem for Eq. cc), inverse column FFT, and the
//                Hermitian step of the complex-to-real row transform -> Y.
//   pair_rows  : inverse row FFT (complex, length Q/2, giving Q reals) of every
//                pair's Y row, rounded to integer joint counts C_AB^{a,b}(chi)
//                (Eq. correlationjointhisto; rounding per Sec. 3.2), fused
//                with the per-shift entropy reduction: the marginals
//                C_A^a = sum_b C_AB^{a,b}, C_B^b = sum_a C_AB^{a,b} and
//                N = sum_a C_A^a (Eq. number), and
//                MI = log2 N + (sum c log2 c (joint) - sum (marginals)) / N,
//                which is Eq. finalentropy + Eq. mientropy rearranged.  The
//                K_A*K_B count maps never reach global memory.
//   peak       : the gamma-gated argmax of Alg. 1 for one map.
#pragma once
#include <type_traits>
#include <cstdint>
#include "common.h"
#include <cooperative_groups.h>
#include "fft.cuh"

namespace cmif {

// ---------------------------------------------------------------------------
// c * log2(c) for an exact non-negative integer c < 2^23 held in a float, in
// fixed point (units of 2^-kFixBits) so that per-shift sums are exact, order
// independent and cheap (integer adds): c * L(c), where for c = m * 2^e,
// m in [1, 2), L(c) = e * 2^F + round(log2(m) * 2^F).  log2(m) comes from the
// MUFU lg2 approximation; the rounding to the 2^-F grid adds at most 2^-(F+1).
// The largest |L(c) 2^-F - log2 c| over every count the epilogue can meet is
// measured exhaustively through cmif_entropy_terms (include/cmif.h).
//
// The sums take c * (L(c) + kTermBias): the bias drops out of every result, because
// each of the joint, A- and B-marginal counts of a shift sums to N (so MI and NMI
// combine the four sums with the biases N - N - N + N = 0), and leaving it in saves an
// add per count.  c = 0 gives 0 whatever L is (Sec. 3.2: 0 log 0 = 0).  The term is one
// fixed function of c, so equal counts cancel exactly between joint and marginal sums.
constexpr int kTermBias = 0x4B000000;
// log2 of a mantissa in [1, 2): no denormals, so the flush-to-zero form (the default one
// carries a rescaling of denormal inputs, three more instructions per count)
__device__ __forceinline__ float lg2_mantissa(float m) {
    float r;
    asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(m));
    return r;
}
__device__ __forceinline__ long long clog2c_biased(float c) {
    const int ci = __float_as_int(c + 8388608.0f) - 0x4B000000;
    const int bits = __float_as_int(c), mb = (bits & 0x7FFFFF) | 0x3F800000;
    // 2^23 + log2(m) 2^23 lies in [2^23, 2^24], where floats are spaced 1 apart and
    // their bit patterns grow by 1 per unit: the FMA rounds log2(m) 2^23 to the
    // nearest integer and the bits hold it above 0x4B000000 (= kTermBias; no
    // float-to-integer conversion).  bits - mb = e 2^23.
    const int t = __float_as_int(fmaf(lg2_mantissa(__int_as_float(mb)), 8388608.0f, 8388608.0f));
    return (long long)ci * (long long)(bits - mb + t);
}
// Two counts at once: the float adds and the FMA as two-lane instructions.
__device__ __forceinline__ void clog2c_biased2(float2 c, long long& t0, long long& t1) {
    const float2 b = __fadd2_rn(c, make_float2(8388608.0f, 8388608.0f));
    const int x0 = __float_as_int(c.x), x1 = __float_as_int(c.y);
    const int m0 = (x0 & 0x7FFFFF) | 0x3F800000, m1 = (x1 & 0x7FFFFF) | 0x3F800000;
    const float2 l = make_float2(lg2_mantissa(__int_as_float(m0)), lg2_mantissa(__int_as_float(m1)));
    const float2 t = __ffma2_rn(l, make_float2(8388608.0f, 8388608.0f), make_float2(8388608.0f, 8388608.0f));
    t0 = (long long)(__float_as_int(b.x) - 0x4B000000) * (long long)(x0 - m0 + __float_as_int(t.x));
    t1 = (long long)(__float_as_int(b.y) - 0x4B000000) * (long long)(x1 - m1 + __float_as_int(t.y));
}

// (q1 + q2) * 2^-kFixBits as a double, |q2| at most a few ulp of q1 (so the sum of the two
// 24-bit values fits 53 bits), by integer arithmetic: the same value that the double add
// gives, but FP64 instructions run at 1/64 rate and the two conversions, the add and the
// product took 4096 of the about 20000 cycles of a row of 4 label pairs at Q = 2048.
__device__ __forceinline__ double double_sum_scaled(float q1, float q2) {
    const int b = __float_as_int(q1);
    if ((b & 0x7FFFFFFF) == 0) return 0.0;  // q1 = 0: the whole sum is 0
    int e = (b >> 23) & 0xFF;
    long long m = (long long)((b & 0x7FFFFF) | 0x800000) << 29;  // 2^52 <= m < 2^53, q1 = m 2^(e - 127 - 52)
    const float q = b < 0 ? -q2 : q2;
    m += __float2int_rn(q * __int_as_float((306 - e) << 23));     // q2 in units of m's last bit
    if (m < (1LL << 52)) { m <<= 1; --e; }
    if (m >= (1LL << 53)) { m >>= 1; ++e; }
    const unsigned long long r = ((unsigned long long)(e - 127 - kFixBits + 1023) << 52) + (unsigned long long)(m - (1LL << 52));
    return __longlong_as_double((long long)(r | ((unsigned long long)(b < 0) << 63)));
}

// MI(chi) = (S + N log2 N) / N, where S = sum_joint c log2 c - sum_A - sum_B and
// every c log2 c term (N log2 N included) comes from clog2c_biased, so that MI is
// exactly 0 whenever the entropies cancel exactly (e.g. a single label).
__device__ __forceinline__ double mi_finish(long long S, int N) {
    if (N <= 0) return 0.0;  // 0/0 = 0: no overlap, no information (Sec. 3.2)
    const long long Sp = S + clog2c_biased((float)N);
    const float sh = (float)Sp;
    const long long rem = Sp - (long long)sh;
    const float sl = (float)rem;
    const float fN = (float)N;
    const float inv = 1.0f / fN;
    const float q1 = sh * inv;
    const float r1 = fmaf(-q1, fN, sh) + sl;
    const float q2 = r1 * inv;
    return double_sum_scaled(q1, q2);
}

// NMI(chi) = (H_A + H_B) / H_AB (the normalised MI the paper cites next to
// MI, Sec. 2.1), from the same fixed-point sums kept apart: SJ = sum_joint c log2 c,
// SM = sum_A + sum_B.  With T(N) = N log2 N: H_A + H_B = (2 T(N) - SM) / N and
// H_AB = (T(N) - SJ) / N.  0 when N = 0 or H_AB = 0 (0/0 = 0, Sec. 3.2).
__device__ __forceinline__ double nmi_finish(long long SJ, long long SM, int N) {
    if (N <= 0) return 0.0;
    const long long TN = clog2c_biased((float)N);
    const long long den = TN - SJ;
    if (den == 0) return 0.0;
    return (double)(2 * TN - SM) / (double)den;
}

// Per-position entropy sums of the row epilogue: MI keeps one signed sum
// (joint terms in, marginal terms out); NMI keeps the two apart.
template <bool NMI>
struct EntAcc;
template <>
struct EntAcc<false> {
    long long s;
    __device__ __forceinline__ void zero() { s = 0; }
    __device__ __forceinline__ void joint(long long t) { s += t; }
    __device__ __forceinline__ void marg(long long t) { s -= t; }
    __device__ __forceinline__ void add(const EntAcc& o) { s += o.s; }
    __device__ __forceinline__ double finish(int N) const { return mi_finish(s, N); }
};
template <>
struct EntAcc<true> {
    long long j, m;
    __device__ __forceinline__ void zero() { j = 0; m = 0; }
    __device__ __forceinline__ void joint(long long t) { j += t; }
    __device__ __forceinline__ void marg(long long t) { m += t; }
    __device__ __forceinline__ void add(const EntAcc& o) { j += o.j; m += o.m; }
    __device__ __forceinline__ double finish(int N) const { return nmi_finish(j, m, N); }
};

__device__ __forceinline__ void atomic_max_float_pos(unsigned* addr, float v) {
    atomicMax(addr, __float_as_uint(v));  // v >= 0: float order = unsigned order
}

// A pre-rounding count -> the count as a float, and its residual; modular counts are exact.
template <typename T>
__device__ __forceinline__ float round_count(T v, float& res) {
    if constexpr (std::is_same<T, m31>::value) {
        return m31_count(v);
    } else {
        const float c = rintf(v);
        res = fmaxf(res, fabsf(v - c));
        return c;
    }
}

// Map a circular shift index (0..n-1) to the output map index, or -1 when the
// shift lies in the zero-padding gap (cannot happen for in-range shifts).
__device__ __forceinline__ int circ_to_out(int s, int n, int lo_count /*H_A or W_A*/, int hi_max /*H_B-1*/) {
    if (s <= hi_max) return s + lo_count - 1;
    if (s >= n - (lo_count - 1)) return s - n + lo_count - 1;
    return -1;
}

// ---------------------------------------------------------------------------
// Team geometry for a transform of length N in precision T.
__host__ __device__ constexpr int pow2_floor(int n) { return n < 2 ? 1 : 2 * pow2_floor(n / 2); }

// MMAX caps the lanes per group (and the values per lane): the default is the
// register budget of T; a smaller one trades a radix-R step for more warps.
template <typename T, int N, int MMAX = max_m<T>()>
struct TeamGeom {
    static constexpr int M = team_m(N, MMAX);
    static constexpr int R = N / (M * M);
    static constexpr int TEAM = R * M;                                        // lanes
    static constexpr int SCRATCH = team_scratch_bytes<T, M, R>();            // bytes of FFT scratch
};

// ---------------------------------------------------------------------------
// Forward row transforms.  Block = (row y, TPB plane pairs); team t takes the
// plane pair pp = blockIdx.y * TPB + t (planes 2pp, 2pp+1).  The block first
// stages the row as one byte per pixel (the label, or kMaskedOut where the
// mask is 0; the label range is checked here), then every team builds its two
// level sets from shared memory.  With a weight image WX (spatially weighted
// MI, Sec. 3.3) the level sets carry the weight W(x) instead of 1 (weight 0 plays
// the mask's 0) and the row's weights are staged too.
constexpr unsigned char kMaskedOut = 255;

template <typename T, int Q>
struct FwdRowsCfg {
    using G = TeamGeom<T, Q>;
    static constexpr int M = G::M, R = G::R, TEAM = G::TEAM;
    // residues: small blocks, so that a launch that needs few planes (CMIF_AUTO's second
    // precision) still fills the SMs: one label pair of 1024^2, Q = 2048: 141 us at 256 threads
    static constexpr int TARGET = std::is_same<T, m31>::value ? 64 : 256;
    static constexpr int TPB = TEAM >= TARGET ? 1 : TARGET / TEAM;
    static constexpr int THREADS = TPB * TEAM;
    static constexpr int MIN_BLOCKS = sizeof(T) == 4 && THREADS <= 512 ? 512 / THREADS : 1;
    static constexpr int REGION = (int)(Q * sizeof(cpx<T>)) > G::SCRATCH ? (int)(Q * sizeof(cpx<T>)) : G::SCRATCH;
    static constexpr size_t smem(int W, bool weighted) {
        return (size_t)TPB * REGION + (((size_t)W + 15) & ~(size_t)15) + (weighted ? (size_t)W * sizeof(double) : 0);
    }
};

template <typename T, int Q>
__global__ void __launch_bounds__(FwdRowsCfg<T, Q>::THREADS, FwdRowsCfg<T, Q>::MIN_BLOCKS)
k_fwd_rows(const int32_t* __restrict__ X, const uint8_t* __restrict__ MX, const double* __restrict__ WX, int H, int W,
           int K, int Qs, cpx<T>* __restrict__ T1, Tw<T> tw, DevStatus* __restrict__ st, int conditional,
           int* __restrict__ popc, const unsigned char* __restrict__ plane_need) {
    // popc (nullable): per-label pixel counts under mask 1 are added to popc[0 .. K).
    // plane_need (nullable): only planes whose entry is 1 are transformed (a team
    // whose two planes are both unneeded idles; a block with no needed plane returns).
    using C = FwdRowsCfg<T, Q>;
    if (conditional && !(st->flags & STATUS_ESCALATE)) return;
    constexpr int M = C::M, R = C::R;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    unsigned char* code = smem_raw + (size_t)C::TPB * C::REGION;
    double* wts = reinterpret_cast<double*>(code + (((size_t)W + 15) & ~(size_t)15));
    const int team = threadIdx.x / C::TEAM, lt = threadIdx.x % C::TEAM, r = lt / M, j = lt % M;
    const int npp = (K + 1) / 2;
    const int y = blockIdx.x, pp = blockIdx.y * C::TPB + team;
    auto needed = [&](int q) {
        if (q >= npp) return false;
        if (!plane_need) return true;
        return plane_need[2 * q] == 1 || (2 * q + 1 < K && plane_need[2 * q + 1] == 1);
    };
    if (plane_need) {
        bool any = false;
        for (int t = 0; t < C::TPB; ++t) any |= needed(blockIdx.y * C::TPB + t);
        if (!any) return;  // uniform over the block
    }
    const bool active = needed(pp);
    const int la = 2 * pp, lb = 2 * pp + 1;
    const int32_t* xr = X + (size_t)y * W;
    const uint8_t* mr = MX ? MX + (size_t)y * W : nullptr;
    bool bad = false;
    // weighted maps run with FP64 transforms only: the other precisions never read weights
    const double* wr = std::is_same<T, double>::value && WX ? WX + (size_t)y * W : nullptr;
    for (int x = threadIdx.x; x < W; x += C::THREADS) {
        const int lab = __ldg(xr + x);
        bool m = mr ? (__ldg(mr + x) != 0) : true;
        if (wr) {
            const double w = __ldg(wr + x);
            m = w > 0.0;
            wts[x] = w;
        }
        if (m && (lab < 0 || lab >= K)) bad = true;
        code[x] = m && lab >= 0 && lab < K ? (unsigned char)lab : kMaskedOut;
    }
    if (bad && blockIdx.y == 0) atomicOr(&st->flags, STATUS_LABEL_RANGE);
    __syncthreads();
    if (popc && blockIdx.y == 0) {
        // label histogram of the row (shared-memory bins in the first team's region,
        // which the transform below only overwrites after the next barrier)
        int* hist = reinterpret_cast<int*>(smem_raw);
        for (int k = threadIdx.x; k < K; k += C::THREADS) hist[k] = 0;
        __syncthreads();
        for (int x = threadIdx.x; x < W; x += C::THREADS) {
            const int c = code[x];
            if (c != kMaskedOut) atomicAdd(&hist[c], 1);
        }
        __syncthreads();
        for (int k = threadIdx.x; k < K; k += C::THREADS)
            if (hist[k]) atomicAdd(&popc[k], hist[k]);
        __syncthreads();
    }
    unsigned char* region = smem_raw + (size_t)team * C::REGION;
    cpx<T>* sm = reinterpret_cast<cpx<T>*>(region);
    auto load = [&](int x) -> cpx<T> {
        if (!active || x >= W) return {T(0), T(0)};
        const int c = code[x];
        T one = T(1);
        if constexpr (std::is_same<T, double>::value) {
            if (wr) one = wts[x];
        }
        return {c == la ? one : T(0), c == lb ? one : T(0)};
    };
    cpx<T> v[M];
    // teams of whole warps without block barriers in their transform: an unneeded one skips it
    const bool run = active || C::TEAM < 32 || R > 2;
    if (run) team_fft<M, R, -1>(v, r, j, load, region + r * grp_scratch_bytes<T, M>(), tw.sq[ilog2c(M)], tw_of<Q>(tw));
    __syncthreads();
    if (run) {
#pragma unroll
        for (int k2 = 0; k2 < M; ++k2) sm[R * (j + M * k2) + r] = v[brev(k2, M)];
    }
    __syncthreads();
    if (!active) return;
    for (int k = lt; k <= Q / 2; k += C::TEAM) {
        const cpx<T> a = sm[k], b = sm[k == 0 ? 0 : Q - k];
        // F_la = (X[k] + conj X[-k]) / 2,  F_lb = (X[k] - conj X[-k]) / (2i)
        T1[((size_t)la * H + y) * Qs + k] = {halve(a.x + b.x), halve(a.y - b.y)};
        if (lb < K) T1[((size_t)lb * H + y) * Qs + k] = {halve(a.y + b.y), halve(b.x - a.x)};
    }
}

// ---------------------------------------------------------------------------
// Forward column transforms.  Item = (TPB adjacent kx columns, plane).  The
// block first stages the item's H x TPB input tile in shared memory with coalesced
// 16-byte loads (column slots XOR-swizzled by row, so that the teams' column
// reads meet few bank conflicts), then each team transforms one column.  FP32: persistent
// blocks; the next item's tile is copied asynchronously (cp.async) into the same buffer from the
// moment the columns are in registers, behind the transform and its stores: with one item per
// block, waiting for the tile (4.1 of 12 cycles per issue) and for the block's other warps (3.7)
// bounded the kernel.  16 labels, us: 1024 x 1024 223 -> 193, 512 x 512 43 -> 38, 32 labels of
// 834 x 834 416 -> 364; P = 768, 331 x 1203, 12 labels 112 -> 77.
template <typename T, int P, int MMAX = max_m<T>()>
struct ColCfg {
    using G = TeamGeom<T, P, MMAX>;
    static constexpr int M = G::M, R = G::R, TEAM = G::TEAM;
    static constexpr int TPB = TEAM >= 256 ? 1 : pow2_floor(256 / TEAM);  // a power of two (swizzle)
    static constexpr int THREADS = TPB * TEAM;
    static constexpr int SWZ = TPB >= 16 ? 0 : (TPB == 8 ? 1 : (TPB == 4 ? 2 : 3));
    static constexpr size_t SCR = (size_t)TPB * G::SCRATCH;
    static constexpr size_t TILE_MAX = (size_t)P * TPB * sizeof(cpx<T>);  // H <= P rows
    static constexpr size_t smem(int H) { return SCR + (size_t)H * TPB * sizeof(cpx<T>); }
    static constexpr bool PIPE = std::is_same<T, float>::value && TPB >= 2;
    // Resident blocks the registers are bounded for (FP32): without spills.  M = 32: two blocks 193 us, three
    // with spills 221 (16 labels, 1024 x 1024).
    static constexpr int f32_blocks() { return M == 32 ? 2 : M == 16 ? (THREADS < 256 ? 4 : 3) : M == 8 ? (THREADS < 256 ? 6 : 4) : 3; }
    static constexpr int MIN_BLOCKS = sizeof(T) == 4 && THREADS <= 256 ? (std::is_same<T, float>::value ? f32_blocks() : 2) : 1;
};

// FP32 groups of 8 lanes and more keep the spectra in the order the packed DFTs take them:
// samples i = 4q .. 4q + 3 of lane j as 8 floats (re, re', im, im' of 4q, 4q + 1, then of
// 4q + 2, 4q + 3) at complex offset (q M + j) 4 of the group.
template <typename T, int M>
__host__ __device__ constexpr bool packed_spectra() { return std::is_same<T, float>::value && M >= 8; }
__device__ __forceinline__ void st_global_32B(void* dst, const float (&v)[8]) {
    asm volatile("st.global.v8.f32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(dst), "f"(v[0]), "f"(v[1]), "f"(v[2]),
                 "f"(v[3]), "f"(v[4]), "f"(v[5]), "f"(v[6]), "f"(v[7]) : "memory");
}

template <typename T, int P, int MMAX>
__global__ void __launch_bounds__(ColCfg<T, P, MMAX>::THREADS, ColCfg<T, P, MMAX>::MIN_BLOCKS)
k_fwd_cols(const cpx<T>* __restrict__ T1, int H, int nplanes, int Qh, int Qs, cpx<T>* __restrict__ F, Tw<T> tw,
           const DevStatus* __restrict__ st, int conditional, T out_scale,
           const unsigned char* __restrict__ plane_need, int slices) {
    // plane_need (nullable): only the planes of labels whose entry is 1 are
    // transformed; plane p belongs to label p / slices (volumes: slices = depth).
    using C = ColCfg<T, P, MMAX>;
    if (conditional && !(st->flags & STATUS_ESCALATE)) return;
    constexpr int M = C::M, R = C::R, TPB = C::TPB;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    cpx<T>* tile = reinterpret_cast<cpx<T>*>(smem_raw + C::SCR);
    const int team = threadIdx.x / C::TEAM, lt = threadIdx.x % C::TEAM, r = lt / M, j = lt % M;
    const int nkxb = (Qh + TPB - 1) / TPB, n_items = nkxb * nplanes;
    auto needed = [&](int it) {  // the next item from `it` on whose plane is needed
        if (plane_need)
            while (it < n_items && plane_need[it / nkxb / slices] != 1) it += gridDim.x;
        return it;
    };
    // Slot of (row y, column c) in the tile: 16-byte pieces of two columns XOR-permuted by the row
    // (without the asynchronous copies, the two columns of a piece, too).
    auto slot = [&](int y, int c) {
        const int sw = (y >> C::SWZ) & (TPB - 1);
        return y * TPB + (c ^ (C::PIPE ? sw & ~1 : sw));
    };
    auto stage = [&](int it) {
        const int plane = it / nkxb, kx0 = (it - plane * nkxb) * TPB;
        const cpx<T>* src = T1 + (size_t)plane * H * Qs + kx0;
        if constexpr (sizeof(T) == 4 && TPB >= 2) {
            // 16-byte pieces (two columns each); Qs and kx0 are even, so a piece is
            // wholly inside the row or wholly beyond Qs (never read: zeros)
            constexpr int PPR = TPB / 2;
            for (int q = threadIdx.x; q < H * PPR; q += C::THREADS) {
                const int y = q / PPR, h = q % PPR;
                const bool in = kx0 + 2 * h < Qs;
                if constexpr (C::PIPE) {
                    const uint32_t dst = (uint32_t)__cvta_generic_to_shared(tile + slot(y, 2 * h));
                    const cpx<T>* from = in ? src + (size_t)y * Qs + 2 * h : T1;
                    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(from), "r"(in ? 16 : 0) : "memory");
                } else {
                    float4 pv = make_float4(0.f, 0.f, 0.f, 0.f);
                    if (in) pv = __ldg(reinterpret_cast<const float4*>(src + (size_t)y * Qs) + h);
                    const int sw = (y >> C::SWZ) & (TPB - 1);
                    if (sw & 1) pv = make_float4(pv.z, pv.w, pv.x, pv.y);
                    reinterpret_cast<float4*>(tile)[y * PPR + (h ^ (sw >> 1))] = pv;
                }
            }
        } else {
            for (int q = threadIdx.x; q < H * TPB; q += C::THREADS) {
                const int y = q / TPB, c = q % TPB;
                tile[slot(y, c)] = kx0 + c < Qs ? src[(size_t)y * Qs + c] : cpx<T>{T(0), T(0)};
            }
        }
    };
    int it = needed(blockIdx.x);
    if (it >= n_items) return;
    stage(it);
    while (true) {
        if constexpr (C::PIPE) asm volatile("cp.async.wait_all;" ::: "memory");
        __syncthreads();
        const int plane = it / nkxb, kx = (it - plane * nkxb) * TPB + team;
        const bool active = kx < Qh;
        const int next = C::PIPE ? needed(it + gridDim.x) : n_items;
        auto load = [&](int y) -> cpx<T> {
            if (!active || y >= H) return {T(0), T(0)};
            return tile[slot(y, team)];
        };
        auto loaded = [&](bool sync) {  // the tile's values are in registers
            if (!C::PIPE || next >= n_items) return;
            if (!sync) __syncthreads();
            stage(next);
        };
        cpx<T> v[M];
        team_fft<M, R, -1>(v, r, j, load, smem_raw + (size_t)team * C::G::SCRATCH + r * grp_scratch_bytes<T, M>(),
                           tw.sq[ilog2c(M)], tw_of<P>(tw), loaded);
        // Column ky is stored at slot (ky % R) * M*M + ky / R: the samples that one
        // group of the pair-product transform (same P, same R) takes are contiguous.
        cpx<T>* out = F + ((size_t)plane * Qh + kx) * P + r * (M * M);
        if (active) {
            if constexpr (packed_spectra<T, M>()) {
#pragma unroll
                for (int q = 0; q < M / 4; ++q) {
                    float w[8];
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        const cpx<T> z = v[brev(4 * q + i, M)];
                        w[4 * (i / 2) + i % 2] = z.x * out_scale;
                        w[4 * (i / 2) + 2 + i % 2] = z.y * out_scale;
                    }
                    st_global_32B(out + 4 * (M * q + j), w);
                }
            } else {
#pragma unroll
                for (int k2 = 0; k2 < M; ++k2) {
                    const cpx<T> z = v[brev(k2, M)];
                    out[j + M * k2] = {z.x * out_scale, z.y * out_scale};
                }
            }
        }
        it = next;
        if (it >= n_items) break;
    }
}

// Read-only loads of complex values through the non-coherent path.
__device__ __forceinline__ cpx<float> __ldg(const cpx<float>* p) {
    const float2 v = ::__ldg(reinterpret_cast<const float2*>(p));
    return {v.x, v.y};
}
__device__ __forceinline__ cpx<double> __ldg(const cpx<double>* p) {
    const double2 v = ::__ldg(reinterpret_cast<const double2*>(p));
    return {v.x, v.y};
}
__device__ __forceinline__ cpx<m31> __ldg(const cpx<m31>* p) {
    const uint2 v = ::__ldg(reinterpret_cast<const uint2*>(p));
    return {m31_of(v.x), m31_of(v.y)};
}

// ---------------------------------------------------------------------------
// Copy n twiddles from global to shared memory (whole block).
template <typename T>
__device__ __forceinline__ void stage_table(cpx<T>* dst, const cpx<T>* __restrict__ src, int n) {
    for (int i = threadIdx.x; i < n; i += blockDim.x) dst[i] = src[i];
}

// ---------------------------------------------------------------------------
// Layout of Y.  A row of Y holds the L = Q/2 inputs z_k of the complex row transform,
// z[m] = x[2m] + i x[2m + 1] = IDFT_L(z_k):
//     z_k = E + i O,  E = y_k + conj(y_{L-k}),  O = (y_k - conj(y_{L-k})) e^{2 pi i k / Q}
// (y_k: the column-inverted product at frequency kx = k <= L).  z_k and z_{L-k} need the
// same two columns, so the pair-column kernel, which has them side by side, forms both: the
// row kernels would each load two values and a twiddle per input.  y_0 and y_L are
// real, so one column transform yields both: column 0 carries y_0 + i y_L.
// Columns are kept in 32-byte chunks (whole sectors) that one block writes:
//   FP32, L / 4 chunks of 4: k0, k1 and the mirrors of k1, k0 (L - k; of 0: L / 2), as
//     two 16-byte halves (direct, mirrored), swapped in every other group of 4 chunks
//     so that the row kernels' reads of consecutive k meet no bank conflicts;
//       split rows (Tensor-Memory row kernel): k1 = k0 + 32 with real and imaginary parts
//       grouped, (re, re', im, im'), in the order of the packed row transform's even and
//       odd inputs;
//       else: k0 = 2c, k1 = 2c + 1 as complex values.
//     Four rows' chunks c form a 128-byte line, lines of one row group in the order of c
//     (Y[pair][row / 4][c][row % 4]): the pair-column kernel's lanes, which hold consecutive
//     rows, write whole lines (8 shared-pipe wavefronts per 32 lanes instead of 32), and the
//     row kernels gather a row's chunks (TMA, or 16-byte asynchronous copies).
//   residues mod p: as FP32 at the other Q;
//   FP64, L / 2 chunks of 2: z_c, z_{L-c}; rows contiguous.
template <typename T>
constexpr int kChunk = sizeof(T) == 4 ? 4 : 2;
// Row widths with a Tensor-Memory row kernel; of these, the ones whose rows are always split
// (the others only where that kernel runs: Geom::split).
__host__ __device__ constexpr bool tm_rows(int Q) {
    return Q == 512 || Q == 1024 || Q == 1536 || Q == 2048 || Q == 3072 || Q == 4096;
}
__host__ __device__ constexpr bool always_split(int Q) { return Q == 512 || Q == 1024 || Q == 2048; }
// Rows of one pair in Y, and the element offset of chunk c of a row.
template <typename T>
__host__ __device__ constexpr int y_rows(int Rout) { return sizeof(T) == 4 ? (Rout + 3) / 4 * 4 : Rout; }
template <typename T>
__device__ __forceinline__ size_t y_chunk(int row, int c, int L) {
    if constexpr (sizeof(T) == 4) return (size_t)(row >> 2) * (4 * L) + c * 16 + (row & 3) * 4;
    else return (size_t)row * L + c * 2;
}
__device__ __forceinline__ bool halves_swapped(int c) { return (c >> 2) & 1; }

// First direct column of chunk c (the second is k0 + 32 in split rows, else k0 + 1).
template <typename T>
__device__ __forceinline__ int chunk_k0(int c, bool split) {
    if constexpr (sizeof(T) == 4) return split ? (c >> 5) * 64 + (c & 31) : 2 * c;
    else return c;
}
__device__ __forceinline__ int mirror_k(int k, int L) { return k ? L - k : L / 2; }
// Column (frequency kx) that slot i of chunk c transforms: the chunk's order in memory.
template <typename T>
__device__ __forceinline__ int chunk_col(int c, int i, int L, bool split) {
    if constexpr (sizeof(T) == 4) {
        const int m = halves_swapped(c) ? i ^ 2 : i;
        const int k = chunk_k0<T>(c, split) + (m == 1 || m == 2 ? (split ? 32 : 1) : 0);
        return m < 2 ? k : mirror_k(k, L);
    } else {
        return i ? mirror_k(c, L) : c;
    }
}
// z_k of a row whose chunks lie CS values apart: back to back (a staged row, FP64), or in Y's
// lines of four rows.
template <typename T>
constexpr int kLine = sizeof(T) == 4 ? 4 * kChunk<T> : kChunk<T>;
template <typename T, int Q, bool SPLIT = false, int CS = kChunk<T>>
__device__ __forceinline__ cpx<T> load_z(const cpx<T>* row, int k) {
    constexpr int L = Q / 2;
    const bool mir = k >= L / 2;
    const int kk = k == L / 2 ? 0 : (mir ? L - k : k);  // the direct partner
    if constexpr (sizeof(T) != 4) {
        return row[CS * kk + (mir ? 1 : 0)];
    } else if constexpr (SPLIT) {
        const int c = (kk >> 6) * 32 + (kk & 31), second = (kk >> 5) & 1;
        const int half = (mir ? 1 : 0) ^ (halves_swapped(c) ? 1 : 0), e = mir ? 1 - second : second;
        const float* f = reinterpret_cast<const float*>(row) + c * 2 * CS + half * 4 + e;
        return {f[0], f[2]};
    } else {
        const int c = kk >> 1, half = (mir ? 1 : 0) ^ (halves_swapped(c) ? 1 : 0), e = mir ? 1 - (kk & 1) : kk & 1;
        return row[c * CS + half * 2 + e];
    }
}
// 32-byte global load (sm_100+), past L1: the spectra are shared through L2
__device__ __forceinline__ void ld_global_32B(const float* src, float (&v)[8]) {
    asm("ld.global.nc.L1::no_allocate.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]), "=f"(v[4]), "=f"(v[5]), "=f"(v[6]), "=f"(v[7])
                 : "l"(src));
}
// Store one chunk in memory order; SPLIT groups real and imaginary parts.
template <bool SPLIT>
__device__ __forceinline__ void store_chunk(cpx<float>* dst, const cpx<float> (&z)[4]) {
    float v[8];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        v[4 * h] = z[2 * h].x;
        v[4 * h + (SPLIT ? 2 : 1)] = z[2 * h].y;
        v[4 * h + (SPLIT ? 1 : 2)] = z[2 * h + 1].x;
        v[4 * h + 3] = z[2 * h + 1].y;
    }
    st_global_32B(dst, v);
}
template <bool SPLIT>
__device__ __forceinline__ void store_chunk(cpx<m31>* dst, const cpx<m31> (&z)[4]) {
    float v[8];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        v[2 * i] = __uint_as_float(z[i].x.v);
        v[2 * i + 1] = __uint_as_float(z[i].y.v);
    }
    st_global_32B(dst, v);
}
template <bool SPLIT, typename T>
__device__ __forceinline__ void store_chunk(cpx<T>* dst, const cpx<T> (&z)[2]) {
    dst[0] = z[0];
    dst[1] = z[1];
}
// The Hermitian step: z_k and z_{L-k} from y_k, y_{L-k}; t = e^{-2 pi i k / Q} (table),
// i O = (y_k - conj(y_{L-k})) i conj(t) = d (t.y, t.x), z_{L-k} = conj(E - i O).  Holds for
// every k, so a chunk with swapped halves only takes the mirror's twiddle.
__device__ __forceinline__ void hermitian_step(cpx<float> yk, cpx<float> ym, cpx<float> t, cpx<float>& zk, cpx<float>& zm) {
    const float2 k2 = make_float2(yk.x, yk.y), m2 = make_float2(ym.x, ym.y);
    const float2 e = __ffma2_rn(m2, make_float2(1.f, -1.f), k2), d = __ffma2_rn(m2, make_float2(-1.f, 1.f), k2);
    const cpx<float> io = cmul(cpx<float>{d.x, d.y}, cpx<float>{t.y, t.x});
    zk = {e.x + io.x, e.y + io.y};
    zm = {e.x - io.x, io.y - e.y};
}
template <typename T>
__device__ __forceinline__ void hermitian_step(cpx<T> yk, cpx<T> ym, cpx<T> t, cpx<T>& zk, cpx<T>& zm) {
    const cpx<T> e = {yk.x + ym.x, yk.y - ym.y}, d = {yk.x - ym.x, yk.y + ym.y};
    const cpx<T> io = cmul(d, cpx<T>{t.y, t.x});
    zk = {e.x + io.x, e.y + io.y};
    zm = {e.x - io.x, io.y - e.y};
}

// ---------------------------------------------------------------------------
// Configuration of the pair-product + inverse column kernel (k_pair_cols below):
// TPB columns per block, one team of R x M lanes per column; the block's shared
// memory holds the teams' P sub-transform values each (a group's slice first serves
// as its transpose scratch) and the twiddle tables.
template <typename T, int P, int MMAX = max_m<T>()>
struct PairColsCfg {
    using G = TeamGeom<T, P, MMAX>;
    static constexpr int M = G::M, R = G::R, TEAM = G::TEAM, NQ = M * M;
    // at least 256 threads, and at least one whole chunk of Y columns
    static constexpr int TPB0 = TEAM >= 256 ? 1 : pow2_floor(256 / TEAM);
    static constexpr int TPB = TPB0 >= kChunk<T> ? TPB0 : kChunk<T>;
    static constexpr int THREADS = TPB * TEAM;
    static constexpr int UPR = TPB / kChunk<T>;  // chunks per block and row
    static constexpr size_t MAIN = (size_t)TPB * P * sizeof(cpx<T>);
    static constexpr int TW_N = R == 2 ? P / 2 : (R > 2 ? P : 0);  // combine twiddles W_P^k
    static constexpr size_t SMEM = MAIN + (size_t)(NQ + TW_N) * sizeof(cpx<T>);
    // Resident blocks the registers are bounded for.  FP32, measured in ps per point with
    // 1 / 2 / 3 / 4 blocks: P = 64 - / 3.58 / 3.10 / 3.03, 128 - / 3.31 / 2.92 / 2.76, 192 - / 3.85 /
    // - / 2.94, 256 - / 2.80 / 2.88 / 3.20, 384 4.01 / 4.05 / 3.44 / -, 512 - / 2.82 / 2.83 / 3.01,
    // 768 3.07 / 3.08 / 2.86 / 2.72, 1536 3.44 / 3.59: as many as hold the values of the transform
    // and of the radix-R combine without spilling
    static constexpr int f32_blocks() {
        if (M == 32) return THREADS <= 256 ? 2 : 1;
        if (R == 6) return M == 8 ? 3 : 1;
        if (M == 16) return R == 3 ? 4 : R <= 2 ? 2 : 1;
        return M == 8 ? 4 : 2;
    }
    // Volumes: depth offsets per item.  The depth sum of one offset loads two slice spectra
    // per product; offsets dz .. dz + NDZ - 1 share A's slice and slide over B's, two loads per
    // NDZ products.  40 x 56 x 64, K = 8 (P = 128): 664 us with one offset per item, 463 with four,
    // still waiting for those loads most of all (2.9 cycles per issue; L2 32 %, FMA pipe 45 %).
    static constexpr int NDZ = std::is_same<T, float>::value ? (M == 8 ? 4 : M == 16 && R <= 3 ? 2 : 1) : 1;
    static constexpr int min_blocks(bool vol) { return sizeof(T) != 4 ? 1 : vol && NDZ > 1 ? 2 : f32_blocks(); }
};

// Pair product + inverse column transform of length P = R*M*M.  Persistent
// blocks walk the items (pair, kx block) with pairs varying fastest, so that
// the items in flight at one time read the same few spectrum columns (L2
// reuse).  Decimation in time across the R groups of a team: group r
// transforms the M*M samples ky = R*m + r (every input is loaded and
// multiplied once per team) and leaves its sub-transform in its own slice of the
// block's buffer (which was its transpose scratch, so nothing but warp syncs comes
// before).  After one barrier every thread takes a row residue k of a chunk's columns: it
// joins the R groups' values by the radix-R butterfly, forms the row transform's
// inputs from the columns and their mirrors (the layout of Y above) and stores R rows'
// 32-byte chunks.  An item thus passes shared memory twice (transpose, combine) and takes two
// block barriers.  While the rows leave, the F_a loads of the block's next item are
// already in flight, and
// items at the head of a kx block ask L2 for the spectrum columns of a later one.
// FP32 groups of 8 lanes and more: spectra in the order of the packed DFTs, 32 bytes per
// load (fwd_cols).  work_ctr must be zero at launch.
// VOL (volumes): items are (pair, NDZ depth offsets dz, kx block); the product is
// the sum over the slices z of conj(F_a,z) F_b,z+dz (the 3-D correlation's
// depth sum, taken before the inverse transform, which is linear), and the
// output row of depth offset index dzo is dzo * R2 + (the image's output row).
template <typename T, int P, bool VOL, int MMAX>
__global__ void __launch_bounds__(PairColsCfg<T, P, MMAX>::THREADS, PairColsCfg<T, P, MMAX>::min_blocks(VOL))
k_pair_cols(const cpx<T>* __restrict__ FA, const cpx<T>* __restrict__ FB, int KA, int KB, int Qh, int HA, int HB,
            int Rout, int r0, int r1, cpx<T>* __restrict__ Y, Tw<T> tw, const cpx<T>* __restrict__ twq,
            const DevStatus* __restrict__ st, int conditional, int* __restrict__ work_ctr, int DA, int DB, int R2,
            const int* __restrict__ plist, const int* __restrict__ lrange, int chunk_off, int chunk_cap, int units,
            int split_rows) {
    // twq: the table of e^{-2 pi i k / Q}, Q = 2 (Qh - 1).
    // units > 1 (images only): several floating images (rotation angles) at once;
    // unit u's spectra are F_b plane b * units + u, its output rows u * R2 + (row).
    // List mode (plist non-null): only the pairs plist[lrange[0] + chunk_off + e],
    // e < min(chunk_cap, lrange[1] - lrange[0] - chunk_off), are computed, pair e's
    // rows going to pair slot e of Y.
    using C = PairColsCfg<T, P, MMAX>;
    if (conditional && !(st->flags & STATUS_ESCALATE)) return;
    constexpr int M = C::M, R = C::R, TPB = C::TPB, NQ = C::NQ, CH = kChunk<T>, UPR = C::UPR;
    const int L = Qh - 1;
    const bool split = std::is_same<T, float>::value && split_rows;  // layout of Y's rows
    const int Dz = VOL ? DA + DB - 1 : 1;
    int npairs = KA * KB, lbase = 0;
    if (plist) {
        lbase = lrange[0] + chunk_off;
        npairs = min(lrange[1] - lbase, chunk_cap);
        if (npairs <= 0) return;  // uniform: nothing listed for this launch
    }
    auto real_pair = [&](int e) { return plist ? ::__ldg(plist + lbase + e) : e; };
    constexpr int NDZ = VOL ? C::NDZ : 1;
    const int U = VOL ? (Dz + NDZ - 1) / NDZ : units;  // the middle item dimension: groups of depth offsets or units
    const int nkxb = (L + TPB - 1) / TPB, n_items = npairs * nkxb * U;
    // L2 prefetch distance in kx blocks: the one beyond those that the blocks in flight cover
    // (columns, us, against a fixed 2: rotations of 300 x 300, 8 x 8 labels 2940 -> 2844, four of 134
    // x 343 208 -> 184; 16 x 16 labels: the same)
    const int ahead = max(2, 1 + (int)gridDim.x / npairs);
    extern __shared__ __align__(128) unsigned char smem_raw[];
    __shared__ int s_next[6];  // the next item: whether there is one, e, a, b, kx block, unit / depth offset
    cpx<T>* xbuf = reinterpret_cast<cpx<T>*>(smem_raw);
    cpx<T>* tw_sq = reinterpret_cast<cpx<T>*>(smem_raw + C::MAIN);
    cpx<T>* tw_n = tw_sq + NQ;
    // Items are handed out in order from a counter (zeroed before the launch), so
    // that the items in flight stay within a few kx blocks whatever the blocks' pace.
    // One thread decodes them (the divisions would cost every thread more than its share
    // of the transform's loads).
    // volumes: kx block outermost, then the depth offset (the slices' spectra of one
    // kx block serve every depth offset); units: the unit outermost, so that the
    // items in flight write the rows of few maps and complete their lines in L2
    auto decode = [&](int it) {
        s_next[0] = it < n_items;
        if (it >= n_items) return;
        const int e = it % npairs, rest = it / npairs, pair = real_pair(e), a = pair / KB;
        s_next[1] = e;
        s_next[2] = a;
        s_next[3] = pair - a * KB;
        s_next[4] = VOL ? rest / U : rest % nkxb;
        s_next[5] = VOL ? rest % U : rest / nkxb;
    };
    if (threadIdx.x == 0) decode(atomicAdd(work_ctr, 1));
    stage_table(tw_sq, tw.sq[ilog2c(M)], NQ);
    if (R > 1) stage_table(tw_n, tw_of<P>(tw), C::TW_N);
    __syncthreads();
    bool more = s_next[0] != 0;
    int e = s_next[1], a = s_next[2], b = s_next[3], kxb = s_next[4], dzo = s_next[5];
    __syncthreads();  // s_next is read by every thread before thread 0 decodes the next item into it
    if (!more) return;
    const int team = threadIdx.x / C::TEAM, lt = threadIdx.x % C::TEAM, r = lt / M, j = lt % M;
    cpx<T>* slice = xbuf + (size_t)team * P + r * NQ;  // this group's transpose scratch, then its sub-transform
    // the frequency kx this team transforms for kx block kxb, or -1 beyond the last
    auto column = [&](int kxb, int t) {
        const int s = kxb * TPB + t;
        return s < L ? chunk_col<T>(s / CH, s % CH, L, split) : -1;
    };
    // group r: the samples ky = R*m + r, m = j + M*i, stored contiguously from slot
    // r*NQ (the forward column transform's output order).  conj(F_a) F_b, F_b
    // carrying the 1/(P Q) of the inverse.
    constexpr bool PK = packed_spectra<T, M>();
    constexpr int H = PK ? M / 2 : 1, NV = PK ? M / 4 : 1;  // pairs, 32-byte loads
    cpx<T> v[PK ? 1 : M];
    float2 re[H], im[H];  // PK: the F_a values, then the products, in pairs
    const size_t lane_off = PK ? (size_t)r * NQ + 4 * j : (size_t)r * NQ + j;
    auto load_fa = [&]() {
        if constexpr (VOL) return;  // volumes sum over slices in the item itself
        const int kx = column(kxb, team);
        const cpx<T>* ga = FA + ((size_t)a * Qh + (kx < 0 ? 0 : kx)) * P + lane_off;
        if constexpr (PK) {
#pragma unroll
            for (int q = 0; q < NV; ++q) {
                float w[8];
                ld_global_32B(reinterpret_cast<const float*>(ga + 4 * M * q), w);
                re[2 * q] = make_float2(w[0], w[1]);
                im[2 * q] = make_float2(w[2], w[3]);
                re[2 * q + 1] = make_float2(w[4], w[5]);
                im[2 * q + 1] = make_float2(w[6], w[7]);
            }
        } else {
#pragma unroll
            for (int i = 0; i < M; ++i) v[i] = __ldg(ga + M * i);
        }
    };
    // conj(a) b of pairs
    auto mulc2 = [](float2 ar, float2 ai, float2 br, float2 bi, float2& pr, float2& pi) {
        pr = __ffma2_rn(ai, bi, __fmul2_rn(ar, br));
        const float2 t = __fmul2_rn(ar, bi);
        pi = make_float2(fmaf(-ai.x, br.x, t.x), fmaf(-ai.y, br.y, t.y));
    };
    // (re, im) += w conj(F_a) F_b of one column, w = 1 or (ROT) i
    auto add_product = [&](auto rotc, const cpx<T>* ga, const cpx<T>* gb) {
        constexpr bool ROT = decltype(rotc)::value;
        if constexpr (PK) {
#pragma unroll
            for (int q = 0; q < NV; ++q) {
                float x[8], y[8];
                ld_global_32B(reinterpret_cast<const float*>(ga + 4 * M * q), x);
                ld_global_32B(reinterpret_cast<const float*>(gb + 4 * M * q), y);
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    float2 pr, pi;
                    mulc2(make_float2(x[4 * h], x[4 * h + 1]), make_float2(x[4 * h + 2], x[4 * h + 3]),
                          make_float2(y[4 * h], y[4 * h + 1]), make_float2(y[4 * h + 2], y[4 * h + 3]), pr, pi);
                    re[2 * q + h] = ROT ? subv(re[2 * q + h], pi) : addv(re[2 * q + h], pr);
                    im[2 * q + h] = ROT ? addv(im[2 * q + h], pr) : addv(im[2 * q + h], pi);
                }
            }
        } else {
#pragma unroll
            for (int i = 0; i < M; ++i) {
                const cpx<T> q = cmulc(__ldg(gb + M * i), __ldg(ga + M * i));
                v[i] = ROT ? cpx<T>{v[i].x - q.y, v[i].y + q.x} : v[i] + q;
            }
        }
    };
    load_fa();
    while (true) {
        int next = 0;
        if (threadIdx.x == 0) next = atomicAdd(work_ctr, 1);
        const int kx = column(kxb, team), pair = a * KB + b;
        if (VOL || kx < 0) {
            if constexpr (PK) {
#pragma unroll
                for (int i = 0; i < H; ++i) re[i] = im[i] = make_float2(0.f, 0.f);
            } else {
#pragma unroll
                for (int i = 0; i < M; ++i) v[i] = {T(0), T(0)};
            }
        }
        float2 sre[NDZ > 1 ? NDZ : 1][H], sim[NDZ > 1 ? NDZ : 1][H];  // NDZ > 1: the depth sums of the item's offsets
        if constexpr (VOL && NDZ > 1) {
#pragma unroll
            for (int s = 0; s < NDZ; ++s)
#pragma unroll
                for (int i = 0; i < H; ++i) sre[s][i] = sim[s][i] = make_float2(0.f, 0.f);
            // offsets dz + s, s < NDZ: slice z of A with slices z + dz + s of B, which slide through
            // a ring of NDZ (zero beyond B's slices)
            const int dz = dzo * NDZ - (DA - 1);
            const int za = max(0, -dz - (NDZ - 1)), zb = min(DA, DB - dz);
            const size_t slice_stride = (size_t)Qh * P;
            auto depth_sum = [&](auto rotc, const cpx<T>* ga, const cpx<T>* gb) {
                constexpr bool ROT = decltype(rotc)::value;
#pragma unroll
                for (int q = 0; q < NV; ++q) {
                    float ring[NDZ][8];
                    auto load_b = [&](int s, int zz) {
                        if (zz >= 0 && zz < DB) {
                            ld_global_32B(reinterpret_cast<const float*>(gb + zz * slice_stride + 4 * M * q), ring[s]);
                        } else {
#pragma unroll
                            for (int x = 0; x < 8; ++x) ring[s][x] = 0.f;
                        }
                    };
#pragma unroll
                    for (int s = 1; s < NDZ; ++s) load_b(s, za + dz + s - 1);
#pragma unroll 1
                    for (int z = za; z < zb; ++z) {
                        float w[8];
                        ld_global_32B(reinterpret_cast<const float*>(ga + z * slice_stride + 4 * M * q), w);
#pragma unroll
                        for (int s = 0; s + 1 < NDZ; ++s)
#pragma unroll
                            for (int x = 0; x < 8; ++x) ring[s][x] = ring[s + 1][x];
                        load_b(NDZ - 1, z + dz + NDZ - 1);
#pragma unroll
                        for (int s = 0; s < NDZ; ++s)
#pragma unroll
                            for (int h = 0; h < 2; ++h) {
                                const int i = 2 * q + h;
                                float2 pr, pi;
                                mulc2(make_float2(w[4 * h], w[4 * h + 1]), make_float2(w[4 * h + 2], w[4 * h + 3]),
                                      make_float2(ring[s][4 * h], ring[s][4 * h + 1]),
                                      make_float2(ring[s][4 * h + 2], ring[s][4 * h + 3]), pr, pi);
                                sre[s][i] = ROT ? subv(sre[s][i], pi) : addv(sre[s][i], pr);
                                sim[s][i] = ROT ? addv(sim[s][i], pr) : addv(sim[s][i], pi);
                            }
                    }
                }
            };
            if (kx >= 0) {
                const cpx<T>* ga = FA + ((size_t)a * DA * Qh + kx) * P + lane_off;
                const cpx<T>* gb = FB + ((size_t)b * DB * Qh + kx) * P + lane_off;
                depth_sum(std::false_type{}, ga, gb);
                if (kx == 0) depth_sum(std::true_type{}, ga + (size_t)L * P, gb + (size_t)L * P);
            }
        } else if constexpr (VOL) {
            if (kx >= 0) {
                const int dz = dzo - (DA - 1);
                const int z0 = dz < 0 ? -dz : 0, z1 = DA < DB - dz ? DA : DB - dz;
                for (int z = z0; z < z1; ++z) {
                    const cpx<T>* ga = FA + ((size_t)(a * DA + z) * Qh + kx) * P + lane_off;
                    const cpx<T>* gb = FB + ((size_t)(b * DB + z + dz) * Qh + kx) * P + lane_off;
                    add_product(std::false_type{}, ga, gb);
                    if (kx == 0) add_product(std::true_type{}, ga + (size_t)L * P, gb + (size_t)L * P);
                }
            }
        } else if (kx >= 0) {
            const cpx<T>* gb = FB + ((size_t)(b * units + dzo) * Qh + kx) * P + lane_off;
            if constexpr (PK) {
#pragma unroll
                for (int q = 0; q < NV; ++q) {
                    float y[8];
                    ld_global_32B(reinterpret_cast<const float*>(gb + 4 * M * q), y);
#pragma unroll
                    for (int h = 0; h < 2; ++h)
                        mulc2(re[2 * q + h], im[2 * q + h], make_float2(y[4 * h], y[4 * h + 1]),
                              make_float2(y[4 * h + 2], y[4 * h + 3]), re[2 * q + h], im[2 * q + h]);
                }
            } else {
#pragma unroll
                for (int i = 0; i < M; ++i) v[i] = cmulc(__ldg(gb + M * i), v[i]);
            }
            // column 0 carries y_0 + i y_L
            if (kx == 0) add_product(std::true_type{}, FA + ((size_t)a * Qh + L) * P + lane_off, gb + (size_t)L * P);
        }
        if (!VOL && !plist && pair < KA + KB && (int)threadIdx.x < TPB) {
            // the items of this kx block with pair < K_A + K_B each prefetch one
            // spectrum's columns of kx block kxb + ahead into L2 (one bulk request per column),
            // or of the next unit's first ones
            int kp = kxb + ahead, up = dzo;
            if (kp >= nkxb) {
                kp -= nkxb;
                ++up;
            }
            const int kf = up < U && kp < nkxb ? column(kp, threadIdx.x) : -1;
            if (kf >= 0) {
                const cpx<T>* src = pair < KA ? FA + ((size_t)pair * Qh + kf) * P
                                              : FB + ((size_t)((pair - KA) * units + up) * Qh + kf) * P;
                asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(src), "r"((unsigned)(P * sizeof(cpx<T>)))
                             : "memory");
            }
        }
        // this item's rows below; its successor's fields once they are known
        cpx<T>* yp = Y + (size_t)e * y_rows<T>(Rout) * L;
        const int c0 = kxb * UPR, dz0 = dzo * NDZ;
#pragma unroll 1
        for (int s = 0; s < NDZ; ++s) {
        if (NDZ > 1) {
            if (dz0 + s >= Dz) break;  // uniform
#pragma unroll
            for (int t = 0; t < NDZ; ++t)
#pragma unroll
                for (int i = 0; i < H; ++i) {
                    re[i] = s == t ? sre[t % (NDZ > 1 ? NDZ : 1)][i] : re[i];
                    im[i] = s == t ? sim[t % (NDZ > 1 ? NDZ : 1)][i] : im[i];
                }
        }
        if constexpr (PK) {
            team_core_pk<M, +1, true>(re, im, j, reinterpret_cast<float*>(slice), reinterpret_cast<const float4*>(tw_sq));
#pragma unroll
            for (int k = 0; k < H; ++k) {
                slice[j + M * k] = {re[k].x, im[k].x};
                slice[j + M * (k + H)] = {re[k].y, im[k].y};
            }
        } else {
            team_fft_core<M, +1>(v, j, slice, tw_sq);
#pragma unroll
            for (int k2 = 0; k2 < M; ++k2) slice[j + M * k2] = v[brev(k2, M)];
        }
        const int row_off = (dz0 + s) * R2;
        if (s == 0 && threadIdx.x == 0) decode(next);
        __syncthreads();
        if (s == 0) {
            more = s_next[0] != 0;
            e = s_next[1], a = s_next[2], b = s_next[3], kxb = s_next[4], dzo = s_next[5];
            if (more) load_fa();
        }
        // Rows k + q NQ, q < R, of chunk c: X[k + q NQ] = sum_s w_R^{sq} (W_P^{sk} E_s[k])
        auto emit = [&](auto splitc) {
            constexpr bool SPLIT = decltype(splitc)::value;
            cpx<T> t[CH / 2];  // the Hermitian step's twiddles of the chunk's first columns
            auto load_t = [&](int c) {
#pragma unroll
                for (int i = 0; i < CH / 2; ++i) {
                    const int kc = chunk_col<T>(c, i, L, SPLIT);
                    t[i] = __ldg(twq + kc);
                }
            };
            // chunk by chunk where the threads divide its rows (twiddles loaded once per chunk),
            // else all the block's chunks in one run
            constexpr bool NEST = NQ % C::THREADS == 0 || UPR == 1;
            for (int h0 = 0; h0 < (NEST ? UPR : 1); ++h0) {
            if (NEST) {
                if ((c0 + h0) * CH >= L) break;
                load_t(c0 + h0);
            }
            for (int u = threadIdx.x; u < (NEST ? NQ : NQ * UPR); u += C::THREADS) {
                const int h = NEST ? h0 : u / NQ, k = NEST ? u : u % NQ, c = c0 + h;
                if (!NEST) {
                    if (c * CH >= L) break;
                    load_t(c);
                }
                cpx<T> x[CH][R];
#pragma unroll
                for (int i = 0; i < CH; ++i) {
                    const cpx<T>* src = xbuf + (size_t)(h * CH + i) * P + k;
                    if constexpr (R == 1) {
                        x[i][0] = src[0];
                    } else if constexpr (R == 2) {
                        const cpx<T> e0 = src[0], e1 = cmul(src[NQ], twl<+1>(tw_n, k));
                        x[i][0] = e0 + e1;
                        x[i][1] = e0 - e1;
                    } else {
                        x[i][0] = src[0];
#pragma unroll
                        for (int s = 1; s < R; ++s) x[i][s] = cmul(src[s * NQ], twl<+1>(tw_n, s * k));
                        dft_nat<R, +1>(x[i]);
                    }
                }
#pragma unroll
                for (int q = 0; q < R; ++q) {
                    int orow = circ_to_out(k + q * NQ, P, HA, HB - 1);
                    if constexpr (VOL) {
                        if (orow < 0) continue;
                        orow += row_off;
                    }
                    if (orow < r0 || orow >= r1) continue;
                    if constexpr (!VOL) orow += row_off;  // the unit's rows
                    cpx<T> z[CH];
#pragma unroll
                    for (int i = 0; i < CH / 2; ++i) hermitian_step(x[i][q], x[CH - 1 - i][q], t[i], z[i], z[CH - 1 - i]);
                    if (c == 0) {  // columns 0 (y_0 + i y_L) and L / 2
                        const cpx<T> g0 = x[0][q], yh = x[CH - 1][q];
                        z[0] = {g0.x + g0.y, g0.x - g0.y};
                        z[CH - 1] = {yh.x + yh.x, T(0) - (yh.y + yh.y)};
                    }
                    store_chunk<SPLIT>(yp + y_chunk<T>(orow, c, L), z);
                }
            }
            }
        };
        if constexpr (std::is_same<T, float>::value) {
            if (split) emit(std::true_type{});
            else emit(std::false_type{});
        } else {
            emit(std::false_type{});
        }
        __syncthreads();  // the buffer's reads (and s_next's) done before it is written again
        }
        if (!more) break;
    }
}

template <typename T, int P, int MMAX = max_m<T>()>
constexpr size_t pair_cols_smem() {
    return PairColsCfg<T, P, MMAX>::SMEM;
}

// ---------------------------------------------------------------------------
// Inverse row transform (L = Q/2 complex inputs z_k, Q reals) + fused entropy epilogue.
// One block per output row (grid-stride).  Per round, NT teams transform NT
// pairs (a-major order); each thread then owns fixed shift positions p and
// accumulates, pair by pair, the joint term T(c), the running A-marginal of
// the current label a, and the B-marginal C_B^b(p) (shared or global memory).
// The rounded counts reach the owners through the teams' scratch, in HALVES
// passes: the scratch holds half a row.
// split > 1 (maps with too few rows to fill the GPU, B-marginals in shared memory): a cluster
// of split blocks takes a row, each the pairs of its own labels a; at the end of the row the
// blocks read each other's partial sums and B-marginals (distributed shared memory) and each
// finishes its share of the positions.
template <typename T, int Q>
struct RowCfg {
    static_assert(sizeof(T) == 4, "FP32 values or residues (weighted maps: RowWCfg)");
    static constexpr int L = Q / 2;
    using G = TeamGeom<T, L>;
    static constexpr int M = G::M, R = G::R, TEAM = G::TEAM;
    // one thread per position of a pass (Q / 2), between one warp and 512
    // threads, so that no thread idles in the epilogue; smaller blocks share an SM.
    static constexpr int BT_TARGET = Q / 2 >= 512 ? 512 : (Q / 2 >= 32 ? Q / 2 : 32);
    // as many teams as the target allows, fewer when that lets the threads divide
    // a pass's positions exactly (no idle lanes in the epilogue) at no more than a
    // quarter fewer teams (3072: 4 teams of 96 lanes, 1536: 8 of 48)
    static constexpr int NT0 = TEAM >= BT_TARGET ? 1 : BT_TARGET / TEAM;
    static constexpr int nt_exact(int nt) {
        return nt <= 1 ? 1 : ((Q / 2) % (nt * TEAM) == 0 ? nt : nt_exact(nt - 1));
    }
    static constexpr int NT = nt_exact(NT0) * 4 >= NT0 * 3 ? nt_exact(NT0) : NT0;
    static constexpr int THREADS = NT * TEAM;
    static constexpr int HALVES = 2;
    static constexpr int QH = Q / HALVES;                      // positions per pass
    static constexpr int UH = (QH + THREADS - 1) / THREADS;    // positions per thread per pass
    static constexpr int U = HALVES * UH;
    static constexpr int REGION = G::SCRATCH;                  // >= QH floats
    static constexpr size_t TEAM_SMEM = (size_t)NT * REGION;
    // each team's next Y row (L complex, 16-byte pieces) is copied into a
    // shared-memory buffer by asynchronous copies (cp.async) while the current round
    // computes; the transform then loads its inputs from shared memory
    static constexpr int STAGE_BYTES = L * 8;
    static constexpr size_t OFF_STAGE = (TEAM_SMEM + 15) / 16 * 16;
    static constexpr size_t OFF_CB = OFF_STAGE + (size_t)NT * STAGE_BYTES;  // B-marginals (shared-memory variant)
    static constexpr int MIN_BLOCKS = THREADS < 512 ? 512 / THREADS : 1;  // <= 128 registers
    static_assert(REGION >= QH * 4, "team scratch must hold one pass of rounded counts");
};

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
    return (uint32_t)__cvta_generic_to_shared(p);
}
// 16-byte asynchronous global-to-shared copy (L2 only), its group commit and the
// wait for all of this thread's copies
__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }

template <typename T, int Q, bool CB_SMEM, bool NMI>
__global__ void __launch_bounds__(RowCfg<T, Q>::THREADS, RowCfg<T, Q>::MIN_BLOCKS)
k_pair_rows(const cpx<T>* __restrict__ Y, Geom g, Tw<T> tw, float* __restrict__ cb_global,
            double* __restrict__ mi_map, int32_t* __restrict__ n_map, int32_t* __restrict__ counts,
            DevStatus* __restrict__ st, int prec_slot, int conditional, const int32_t* __restrict__ ov,
            const int* __restrict__ ov_slot, unsigned* __restrict__ pair_res, int split) {
    // ov / ov_slot (nullable): a pair with ov_slot[pair] = s >= 0 takes its counts
    // from ov[s][row][position] (exact counts from the second precision) instead of
    // its own transform, and its residual is not counted.  pair_res (nullable):
    // each pair's largest residual is folded into pair_res[pair].
    using C = RowCfg<T, Q>;
    constexpr int M = C::M, R = C::R, L = C::L, NT = C::NT, U = C::U, UH = C::UH, BT = C::THREADS;
    constexpr int HALVES = C::HALVES, QH = C::QH;
    if (conditional && !(st->flags & STATUS_ESCALATE)) return;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    float* cb = CB_SMEM ? reinterpret_cast<float*>(smem_raw + C::OFF_CB)
                        : cb_global + (size_t)blockIdx.x * g.KB * Q;
    const int tid = threadIdx.x, team = tid / C::TEAM, lt = tid % C::TEAM, r = lt / M, j = lt % M;
    unsigned char* region = smem_raw + (size_t)team * C::REGION;
    const int KA = g.KA, KB = g.KB, npairs = KA * KB, Rout = g.R, Cout = g.C;
    const size_t RC = (size_t)Rout * Cout;
    float res_max = 0.f;
    int row_max_n = 0;

    // tasks: the window's rows of every unit (units > 1: several maps, R2 rows apart)
    const int nr = g.r1 - g.r0, ntask = g.units * nr;
    const int rank = CB_SMEM ? (int)blockIdx.x % split : 0, ntb = (int)gridDim.x / split, task0 = (int)blockIdx.x / split;
    const int alo = rank * KA / split, plo = alo * KB, phi = (rank + 1) * KA / split * KB;  // this block's pairs
    auto task_row = [&](int tk) { return (tk / nr) * g.R2 + g.r0 + tk % nr; };
    // stage: the team's buffer for the Y row of its current pair; the team's lanes
    // copy a row in 16-byte pieces (the rows start on 32-byte boundaries: L is a
    // multiple of 4)
    const cpx<T>* stage = reinterpret_cast<const cpx<T>*>(smem_raw + C::OFF_STAGE + (size_t)team * C::STAGE_BYTES);
    auto stage_issue = [&](int pair_i, int row_i) {
        // half c % 2 of chunk c / 2, whose rows lie 128 bytes apart (layout of Y)
        const char* src = reinterpret_cast<const char*>(Y + (size_t)pair_i * y_rows<T>(Rout) * L + y_chunk<T>(row_i, 0, L));
        const uint32_t dst = smem_u32(stage);
        for (int c = lt; c < C::STAGE_BYTES / 16; c += C::TEAM)
            cp_async16(dst + 16u * c, src + 128 * (c >> 1) + 16 * (c & 1));
        cp_async_commit();
    };
    if (task0 < ntask && plo + team < phi) stage_issue(plo + team, task_row(task0));
    cp_async_wait_all();
    __syncthreads();
    for (int task = task0; task < ntask; task += ntb) {
        const int row = task_row(task);
        EntAcc<NMI> S[U];
        float CA[U];
        int N[U];
#pragma unroll
        for (int u = 0; u < U; ++u) { S[u].zero(); CA[u] = 0.f; N[u] = 0; }
        for (int b = 0; b < KB; ++b)
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int pl = tid + BT * (u % UH), p = (u / UH) * QH + pl;
                if (pl < QH) cb[(size_t)b * Q + p] = 0.f;
            }
        int cur_a[HALVES];
#pragma unroll
        for (int hf = 0; hf < HALVES; ++hf) cur_a[hf] = alo;
        for (int base = plo; base < phi; base += NT) {
            const int pair = base + team;
            const bool act = pair < phi;
            const int ovs = (act && ov_slot) ? ov_slot[pair] : -1;
            cpx<T> v[M];
            auto transform = [&](auto splitc) {
                constexpr bool SPLIT = decltype(splitc)::value;
                auto load = [&](int k) -> cpx<T> { return act ? load_z<T, Q, SPLIT>(stage, k) : cpx<T>{T(0), T(0)}; };
                team_fft<M, R, +1>(v, r, j, load, region + r * grp_scratch_bytes<T, M>(), tw.sq[ilog2c(M)], tw_of<L>(tw));
            };
            // (Geom::split of the other widths: the Tensor-Memory kernel only)
            transform(std::integral_constant<bool, std::is_same<T, float>::value && always_split(Q)>{});
            // round to the nearest integer; track the worst residual (the exactness guard)
            float rp = 0.f;
            float2 cnt[M];
#pragma unroll
            for (int k = 0; k < M; ++k) cnt[k] = make_float2(round_count(v[k].x, rp), round_count(v[k].y, rp));
            if (ovs < 0) res_max = fmaxf(res_max, rp);
            if (pair_res) {  // per-pair residual: reduce over the team's lanes of each warp
                constexpr int WID = C::TEAM < 32 ? C::TEAM : 32;
                float rr = (act && ovs < 0) ? rp : 0.f;
#pragma unroll
                for (int off = WID / 2; off > 0; off >>= 1) rr = fmaxf(rr, __shfl_xor_sync(0xffffffffu, rr, off));
                if (act && ovs < 0 && (lt % WID) == 0) atomic_max_float_pos(&pair_res[pair], rr);
            }
            const int nt = min(NT, phi - base);
            const int a0 = base / KB, b0 = base - a0 * KB;
#pragma unroll
            for (int hf = 0; hf < HALVES; ++hf) {
                __syncthreads();  // all scratch reads (FFT or previous pass) done
                if (hf == 0) {
                    // the staged rows are consumed: copy this team's next row (the next
                    // round of this task, else round 0 of the block's next task)
                    int np = pair + NT, ntk = task;
                    if (np >= phi) { np = plo + team; ntk = task + ntb; }
                    if (np < phi && ntk < ntask) stage_issue(np, task_row(ntk));
                }
                float2* ob = reinterpret_cast<float2*>(region);
#pragma unroll
                for (int k2 = hf * (M / HALVES); k2 < (hf + 1) * (M / HALVES); ++k2) {
                    const int mf = R * (j + M * k2) + r, m = mf - hf * (L / HALVES);
                    if (ovs >= 0) {  // exact counts of positions 2 mf, 2 mf + 1 from the second precision
                        const int2 q = *reinterpret_cast<const int2*>(ov + ((size_t)ovs * Rout + row) * Q + 2 * mf);
                        ob[m] = make_float2((float)q.x, (float)q.y);
                    } else {
                        ob[m] = cnt[brev(k2, M)];
                    }
                }
                __syncthreads();
                // the round's accumulation, compiled twice: with the debug count maps
                // and without (no per-count test of the counts pointer)
                auto accumulate = [&](auto dbg) {
                    constexpr bool DBG = decltype(dbg)::value;
                    int a = a0, b = b0;
                    if constexpr (!CB_SMEM && !DBG && NT * UH <= 16 && C::THREADS <= 384) {  // registers to spare
                        if (nt == NT && NT <= KB) {
                            // the round's pairs have distinct labels b: load their B-marginal
                            // slots (global memory) together, one memory latency per pass
                            // instead of one per pair
                            float cbv[NT][UH];
#pragma unroll
                            for (int t = 0; t < NT; ++t) {
                                const float* cbb = cb + (size_t)b * Q + hf * QH;
#pragma unroll
                                for (int uh = 0; uh < UH; ++uh) {
                                    const int pl = tid + BT * uh;
                                    cbv[t][uh] = pl < QH ? cbb[pl] : 0.f;
                                }
                                if (++b == KB) b = 0;
                            }
                            b = b0;
#pragma unroll
                            for (int t = 0; t < NT; ++t) {
                                if (a != cur_a[hf]) {
#pragma unroll
                                    for (int uh = 0; uh < UH; ++uh) {
                                        const int u = hf * UH + uh, pl = tid + BT * uh;
                                        if (pl >= QH) continue;
                                        S[u].marg(clog2c_biased(CA[u]));
                                        N[u] += (int)CA[u];
                                        CA[u] = 0.f;
                                    }
                                    cur_a[hf] = a;
                                }
                                const float* obt = reinterpret_cast<const float*>(smem_raw + (size_t)t * C::REGION);
                                float* cbb = cb + (size_t)b * Q + hf * QH;
#pragma unroll
                                for (int uh = 0; uh < UH; ++uh) {
                                    const int u = hf * UH + uh, pl = tid + BT * uh;
                                    if (pl >= QH) continue;
                                    const float c = obt[pl];
                                    S[u].joint(clog2c_biased(c));
                                    CA[u] += c;
                                    cbb[pl] = cbv[t][uh] + c;
                                }
                                if (++b == KB) { b = 0; ++a; }
                            }
                            return;
                        }
                    }
                    for (int t = 0; t < nt; ++t) {
                        if (a != cur_a[hf]) {  // uniform: the A-marginal of label cur_a is complete
#pragma unroll
                            for (int uh = 0; uh < UH; ++uh) {
                                const int u = hf * UH + uh, pl = tid + BT * uh;
                                if (pl >= QH) continue;
                                S[u].marg(clog2c_biased(CA[u]));
                                N[u] += (int)CA[u];
                                if constexpr (DBG) {
                                    const int c = circ_to_out(hf * QH + pl, Q, g.WA, g.WB - 1);
                                    if (c >= 0)
                                        counts[((size_t)npairs + cur_a[hf]) * RC + (size_t)row * Cout + c] = (int)CA[u];
                                }
                                CA[u] = 0.f;
                            }
                            cur_a[hf] = a;
                        }
                        const float* obt = reinterpret_cast<const float*>(smem_raw + (size_t)t * C::REGION);
                        float* cbb = cb + (size_t)b * Q + hf * QH;
#pragma unroll
                        for (int uh = 0; uh < UH; ++uh) {
                            const int u = hf * UH + uh, pl = tid + BT * uh;
                            if (pl >= QH) continue;
                            const float c = obt[pl];
                            S[u].joint(clog2c_biased(c));
                            CA[u] += c;
                            cbb[pl] += c;
                            if constexpr (DBG) {
                                const int cc = circ_to_out(hf * QH + pl, Q, g.WA, g.WB - 1);
                                if (cc >= 0) counts[(size_t)(base + t) * RC + (size_t)row * Cout + cc] = (int)c;
                            }
                        }
                        if (++b == KB) { b = 0; ++a; }
                    }
                };
                if (counts) accumulate(std::true_type{});
                else accumulate(std::false_type{});
            }
            cp_async_wait_all();  // the next round's rows, visible after the barrier
            __syncthreads();  // the next round's transforms overwrite the scratch read above
        }
        if constexpr (CB_SMEM) {
            if (split > 1) {
                namespace cg = cooperative_groups;
                const cg::cluster_group cluster = cg::this_cluster();
                EntAcc<NMI>* part_s = reinterpret_cast<EntAcc<NMI>*>(smem_raw + (C::OFF_CB + (size_t)KB * Q * sizeof(float) + 15) / 16 * 16);
                int* part_n = reinterpret_cast<int*>(part_s + Q);
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    const int pl = tid + BT * (u % UH), p = (u / UH) * QH + pl;
                    if (pl >= QH) continue;
                    S[u].marg(clog2c_biased(CA[u]));
                    N[u] += (int)CA[u];
                    const int cidx = circ_to_out(p, Q, g.WA, g.WB - 1);
                    if (counts && cidx >= 0) counts[((size_t)npairs + cur_a[u / UH]) * RC + (size_t)row * Cout + cidx] = (int)CA[u];
                    part_s[p] = S[u];
                    part_n[p] = N[u];
                }
                cluster.sync();
                for (int p = rank * Q / split + tid; p < (rank + 1) * Q / split; p += BT) {
                    EntAcc<NMI> s;
                    s.zero();
                    int n = 0;
                    for (int r2 = 0; r2 < split; ++r2) {
                        s.add(cluster.map_shared_rank(part_s, r2)[p]);
                        n += cluster.map_shared_rank(part_n, r2)[p];
                    }
                    const int cidx = circ_to_out(p, Q, g.WA, g.WB - 1);
                    for (int b = 0; b < KB; ++b) {
                        float c = 0.f;
                        for (int r2 = 0; r2 < split; ++r2) c += cluster.map_shared_rank(cb, r2)[(size_t)b * Q + p];
                        s.marg(clog2c_biased(c));
                        if (counts && cidx >= 0) counts[((size_t)npairs + KA + b) * RC + (size_t)row * Cout + cidx] = (int)c;
                    }
                    if (cidx < 0) continue;
                    const size_t o = (size_t)row * Cout + cidx;
                    mi_map[o] = s.finish(n);
                    if (n_map) n_map[o] = n;
                    if (cidx >= g.c0 && cidx < g.c1) row_max_n = max(row_max_n, n);
                }
                cluster.sync();  // the others' reads of this block's sums are done
                continue;
            }
        }
        // the B-marginals: all of this thread's positions of one label loaded together
        for (int b = 0; b < KB; ++b) {
            float cbv[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int pl = tid + BT * (u % UH), p = (u / UH) * QH + pl;
                cbv[u] = pl < QH ? cb[(size_t)b * Q + p] : 0.f;
            }
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int pl = tid + BT * (u % UH), p = (u / UH) * QH + pl;
                if (pl >= QH) continue;
                S[u].marg(clog2c_biased(cbv[u]));
                if (counts) {
                    const int cidx = circ_to_out(p, Q, g.WA, g.WB - 1);
                    if (cidx >= 0) counts[((size_t)npairs + KA + b) * RC + (size_t)row * Cout + cidx] = (int)cbv[u];
                }
            }
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int pl = tid + BT * (u % UH), p = (u / UH) * QH + pl;
            if (pl >= QH) continue;
            const int cidx = circ_to_out(p, Q, g.WA, g.WB - 1);
            S[u].marg(clog2c_biased(CA[u]));
            N[u] += (int)CA[u];
            if (counts && cidx >= 0) counts[((size_t)npairs + cur_a[u / UH]) * RC + (size_t)row * Cout + cidx] = (int)CA[u];
            if (cidx < 0) continue;
            const size_t o = (size_t)row * Cout + cidx;
            mi_map[o] = S[u].finish(N[u]);
            if (n_map) n_map[o] = N[u];
            if (cidx >= g.c0 && cidx < g.c1) row_max_n = max(row_max_n, N[u]);
        }
        __syncthreads();
    }
    // block reductions of the residual and max N
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        res_max = fmaxf(res_max, __shfl_xor_sync(0xffffffffu, res_max, off));
        row_max_n = max(row_max_n, __shfl_xor_sync(0xffffffffu, row_max_n, off));
    }
    if ((tid & 31) == 0) {
        atomic_max_float_pos(&st->res_bits[prec_slot], res_max);
        atomicMax(&st->max_n, row_max_n);
    }
}

// ---------------------------------------------------------------------------
// Exact counts of listed pairs in the second precision (per-pair escalation of
// CMIF_AUTO): the inverse row transform (complex-to-real, length Q) of rows
// [r0, r1) of the chunk's column-inverted products, rounded to the nearest
// integers (Sec. 3.2).  The counts of list slot s = lrange[0] + chunk_off + e
// (chunk pair e) go to ov[s][row][0 .. Q); the FP32 row kernels then take them
// in place of their own.  The largest residual goes to st->res_bits[1].
template <typename T, int Q>
struct RowCntCfg {
    static constexpr int L = Q / 2;
    using G = TeamGeom<T, L>;
    static constexpr int M = G::M, R = G::R, TEAM = G::TEAM;
    static constexpr int NT = TEAM >= 128 ? 1 : 128 / TEAM;
    static constexpr int THREADS = NT * TEAM;
    static constexpr size_t SMEM = (size_t)NT * G::SCRATCH;
};

template <typename T, int Q>
__global__ void __launch_bounds__(RowCntCfg<T, Q>::THREADS)
k_pair_rows_counts(const cpx<T>* __restrict__ Y, Geom g, Tw<T> tw, const int* __restrict__ lrange, int chunk_off,
                   int chunk_cap, int32_t* __restrict__ ov, DevStatus* __restrict__ st) {
    using C = RowCntCfg<T, Q>;
    constexpr int M = C::M, R = C::R, L = C::L, NT = C::NT;
    const int lbase = lrange[0] + chunk_off;
    const int np = min(lrange[1] - lbase, chunk_cap);
    if (np <= 0) return;  // uniform: nothing listed for this launch
    extern __shared__ __align__(128) unsigned char smem_raw[];
    const int team = threadIdx.x / C::TEAM, lt = threadIdx.x % C::TEAM, r = lt / M, j = lt % M;
    unsigned char* region = smem_raw + (size_t)team * C::G::SCRATCH;
    const int nrows = g.r1 - g.r0;
    const long long ntask = (long long)np * nrows;
    float res = 0.f;
    // a uniform trip count per block: every lane of a warp takes part in each transform's warp syncs
    for (long long t0 = (long long)blockIdx.x * NT; t0 < ntask; t0 += (long long)gridDim.x * NT) {
        const long long t = t0 + team;
        const bool act = t < ntask;
        const int e = act ? (int)(t / nrows) : 0, row = g.r0 + (act ? (int)(t % nrows) : 0);
        const cpx<T>* yr = Y + (size_t)e * y_rows<T>(g.R) * L + y_chunk<T>(row, 0, L);
        auto load = [&](int k) -> cpx<T> { return act ? load_z<T, Q, false, kLine<T>>(yr, k) : cpx<T>{T(0), T(0)}; };
        cpx<T> v[M];
        team_fft<M, R, +1>(v, r, j, load, region + r * grp_scratch_bytes<T, M>(), tw.sq[ilog2c(M)],
                           tw_of<L>(tw));
        if (act) {
            int32_t* o = ov + ((size_t)(lbase + e) * g.R + row) * Q;
#pragma unroll
            for (int k2 = 0; k2 < M; ++k2) {
                const int mf = R * (j + M * k2) + r;
                const cpx<T> z = v[brev(k2, M)];
                *reinterpret_cast<int2*>(o + 2 * mf) = make_int2((int)round_count(z.x, res), (int)round_count(z.y, res));
            }
        }
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) res = fmaxf(res, __shfl_xor_sync(0xffffffffu, res, off));
    if ((threadIdx.x & 31) == 0) atomic_max_float_pos(&st->res_bits[1], res);
}

// ---------------------------------------------------------------------------
// Spatially weighted MI (Sec. 3.3): the inverse row transform of weighted
// correlations (FP64 transforms) and the MI of their real-valued counts.  The
// counts are not integers, so nothing is rounded: each position accumulates
// sum c log2 c over joint, A- and B-marginal counts in FP64, with c log2 c = 0
// for c <= 0 (a count that the transform's rounding error takes below 0).
// MI = (S_joint - S_A - S_B + N log2 N) / N, N = sum_a C_A^a; 0 when N <= 0.
// One block per output row (grid-stride), NT teams transform NT pairs per round
// (a-major order); the B-marginals live in the block's global slice cbw.
template <int Q>
struct RowWCfg {
    static constexpr int L = Q / 2;
    using G = TeamGeom<double, L>;
    static constexpr int M = G::M, R = G::R, TEAM = G::TEAM;
    static constexpr int NT = TEAM >= 256 ? 1 : 256 / TEAM;
    static constexpr int THREADS = NT * TEAM;
    static constexpr int U = (Q + THREADS - 1) / THREADS;  // positions per thread
    static constexpr int REGION = G::SCRATCH;              // one row of Q doubles
    static constexpr size_t OFF_LG = (size_t)NT * REGION;
    static constexpr size_t SMEM = OFF_LG + (size_t)(1 << 9) * 16;  // + the logarithm table
    static_assert(REGION >= Q * 8, "team scratch must hold one row of counts");
};

// log2 c for c > 0, table-driven (Tang, ACM Trans. Math. Software 16(4), 1990): c = m 2^e, the top 9
// bits of m pick r ~ 1 / m with log2(1 / r) tabulated, z = m r - 1 is exact to one rounding,
// |z| <= 2^-9, and log2(1 + z) = (z - z^2/2 + z^3/3 - ...) / ln 2 to z^6 (the rest is below
// 2^-64).  at most 1 ulp (|log2 c| >= 1; 2e-16 absolute below).  Nine FP64 instructions, at 1/64 rate the kernel's scarcest; the math library's log2
// took over half of the kernel's time (200 x 256, K = 12: 3.45 ms, with the table 1.83).
constexpr int kLgBits = 9, kLgSize = 1 << kLgBits;
__device__ __forceinline__ double lg2_table(double c, const double2* lg) {
    const int hi = __double2hiint(c);
    if (hi < 0x00100000) return log2(c);  // denormal
    const double2 t = lg[(hi >> (20 - kLgBits)) & (kLgSize - 1)];
    const double m = __hiloint2double((hi & 0xFFFFF) | 0x3FF00000, __double2loint(c));
    const double z = fma(m, t.x, -1.0);
    // e as a double: 2^52 + 2^31 + e, less 2^52 + 2^31
    const double e = __hiloint2double(0x43300000, ((hi >> 20) - 1023) ^ (int)0x80000000) - 4503601774854144.0;
    constexpr double il = 1.4426950408889634074;  // 1 / ln 2
    double p = fma(z, -il / 6, il / 5);
    p = fma(z, p, -il / 4);
    p = fma(z, p, il / 3);
    p = fma(z, p, -il / 2);
    p = fma(z, p, il);
    return e + fma(z, p, t.y);
}
__device__ __forceinline__ double xlog2x(double c, const double2* lg) { return c > 0.0 ? c * lg2_table(c, lg) : 0.0; }

template <int Q>
__global__ void __launch_bounds__(RowWCfg<Q>::THREADS, 1)
k_pair_rows_w(const cpx<double>* __restrict__ Y, Geom g, Tw<double> tw, double* __restrict__ cbw,
              double* __restrict__ mi_map, double* __restrict__ nw_map, DevStatus* __restrict__ st) {
    using C = RowWCfg<Q>;
    constexpr int M = C::M, R = C::R, L = C::L, NT = C::NT, U = C::U, BT = C::THREADS;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    const int tid = threadIdx.x, team = tid / C::TEAM, lt = tid % C::TEAM, r = lt / M, j = lt % M;
    unsigned char* region = smem_raw + (size_t)team * C::REGION;
    double2* lg = reinterpret_cast<double2*>(smem_raw + C::OFF_LG);
    for (int i = tid; i < kLgSize; i += BT) lg[i] = tw.lg[i];  // visible after the first round's barriers
    const int KB = g.KB, npairs = g.KA * g.KB, Rout = g.R, Cout = g.C;
    double* cb = cbw + (size_t)blockIdx.x * KB * Q;
    double row_max_n = 0.0;
    for (int row = g.r0 + blockIdx.x; row < g.r1; row += gridDim.x) {
        double S[U], CA[U], N[U];
#pragma unroll
        for (int u = 0; u < U; ++u) { S[u] = 0.0; CA[u] = 0.0; N[u] = 0.0; }
        for (int b = 0; b < KB; ++b)
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int p = tid + BT * u;
                if (p < Q) cb[(size_t)b * Q + p] = 0.0;
            }
        int cur_a = 0;
        for (int base = 0; base < npairs; base += NT) {
            const int pair = base + team;
            const bool act = pair < npairs;
            const cpx<double>* yr = Y + ((size_t)(act ? pair : 0) * Rout + row) * L;
            auto load = [&](int k) -> cpx<double> { return act ? load_z<double, Q>(yr, k) : cpx<double>{0.0, 0.0}; };
            cpx<double> v[M];
            team_fft<M, R, +1>(v, r, j, load, region + r * grp_scratch_bytes<double, M>(), tw.sq[ilog2c(M)],
                               tw_of<L>(tw));
            __syncthreads();  // all transforms done with their scratch
            double2* ob = reinterpret_cast<double2*>(region);
#pragma unroll
            for (int k2 = 0; k2 < M; ++k2) {
                const cpx<double> z = v[brev(k2, M)];
                ob[R * (j + M * k2) + r] = make_double2(z.x, z.y);  // positions 2m, 2m + 1
            }
            __syncthreads();
            const int nt = min(NT, npairs - base);
            int a = base / KB, b = base - (base / KB) * KB;
            for (int t = 0; t < nt; ++t) {
                if (a != cur_a) {  // uniform: the A-marginal of label cur_a is complete
#pragma unroll
                    for (int u = 0; u < U; ++u) {
                        S[u] -= xlog2x(CA[u], lg);
                        N[u] += CA[u];
                        CA[u] = 0.0;
                    }
                    cur_a = a;
                }
                const double* obt = reinterpret_cast<const double*>(smem_raw + (size_t)t * C::REGION);
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    const int p = tid + BT * u;
                    if (p >= Q) continue;
                    const double c = fmax(obt[p], 0.0);
                    S[u] += xlog2x(c, lg);
                    CA[u] += c;
                    cb[(size_t)b * Q + p] += c;
                }
                if (++b == KB) { b = 0; ++a; }
            }
            __syncthreads();  // the next round's transforms overwrite the scratch read above
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int p = tid + BT * u;
            if (p >= Q) continue;
            S[u] -= xlog2x(CA[u], lg);
            N[u] += CA[u];
            for (int b = 0; b < KB; ++b) S[u] -= xlog2x(cb[(size_t)b * Q + p], lg);
            const int cidx = circ_to_out(p, Q, g.WA, g.WB - 1);
            if (cidx < 0) continue;
            const size_t o = (size_t)row * Cout + cidx;
            mi_map[o] = N[u] > 0.0 ? (S[u] + xlog2x(N[u], lg)) / N[u] : 0.0;
            nw_map[o] = N[u];
            if (cidx >= g.c0 && cidx < g.c1) row_max_n = fmax(row_max_n, N[u]);
        }
        __syncthreads();
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) row_max_n = fmax(row_max_n, __shfl_xor_sync(0xffffffffu, row_max_n, off));
    if ((tid & 31) == 0) atomicMax(&st->max_nw_bits, (unsigned long long)__double_as_longlong(row_max_n));
}

template <typename T, int Q>
constexpr size_t pair_rows_smem(int KB, bool cb_smem) {
    return RowCfg<T, Q>::OFF_CB + (cb_smem ? (size_t)KB * Q * sizeof(float) : 0);
}

// ---------------------------------------------------------------------------
// gamma-gated argmax of Alg. 1 over one map: N_cal = gamma * max N; best MI
// among shifts with N >= N_cal; ties to the lowest map index.
struct PeakPart {
    double mi;
    long long idx;
};



}  // namespace cmif
