// Register / shared-memory FFT building blocks for the CMIF transforms.
//
// The paper computes every cross-correlation of Eq. correlationjointhisto
// in the frequency domain with FFTs (Sec. 3.5, Eq. maincomplexity).  These
// are the transforms, written for sm_103a:
//
//  * dft_reg<M>     : an M-point DFT held in one thread's registers, radix-2
//                     decimation in frequency, twiddles folded to compile-time
//                     constants.  Output in bit-reversed register order.  FP32
//                     DFTs of 8 and more points are the packed ones of fft_pk.cuh.
//  * team_fft<M,R>  : a length N = R*M*M DFT done by a "team" of R groups of
//                     M lanes (M points per lane).  The four-step split
//                     N' = M*M needs a single shared-memory transpose (XOR
//                     swizzled, conflict-free); R > 1 adds a radix-R
//                     decimation-in-frequency pre-step fused into the loads,
//                     so group r produces the outputs k = r (mod R).
//
// Sign convention: DIR = -1 is the forward transform X[k] = sum x[n] e^{-2 pi i kn/N},
// DIR = +1 the unnormalised inverse.
#pragma once
#include <cstdint>
#include <type_traits>
#include <cuda_runtime.h>
#include "m31.cuh"

namespace cmif {

template <typename T>
struct cpx {
    T x, y;
};

template <typename T>
__device__ __forceinline__ cpx<T> operator+(cpx<T> a, cpx<T> b) { return {a.x + b.x, a.y + b.y}; }
template <typename T>
__device__ __forceinline__ cpx<T> operator-(cpx<T> a, cpx<T> b) { return {a.x - b.x, a.y - b.y}; }
// FP32: one packed two-lane instruction per complex add / subtract (sm_100+
// FADD2 / FFMA2; each lane rounds like the scalar op, a - b as fma(b, -1, a)).
__device__ __forceinline__ cpx<float> operator+(cpx<float> a, cpx<float> b) {
    const float2 r = __fadd2_rn(make_float2(a.x, a.y), make_float2(b.x, b.y));
    return {r.x, r.y};
}
__device__ __forceinline__ cpx<float> operator-(cpx<float> a, cpx<float> b) {
    const float2 r = __ffma2_rn(make_float2(b.x, b.y), make_float2(-1.f, -1.f), make_float2(a.x, a.y));
    return {r.x, r.y};
}
template <typename T>
__device__ __forceinline__ cpx<T> cmul(cpx<T> a, cpx<T> b) {
    return {a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x};
}
// a * conj(b)
template <typename T>
__device__ __forceinline__ cpx<T> cmulc(cpx<T> a, cpx<T> b) {
    return {a.x * b.x + a.y * b.y, a.y * b.x - a.x * b.y};
}
// multiply by e^{DIR * i * theta} given (cos theta, sin theta)
template <int DIR, typename T>
__device__ __forceinline__ cpx<T> rot(cpx<T> a, T c, T s) {
    if (DIR < 0) return {a.x * c + a.y * s, a.y * c - a.x * s};
    return {a.x * c - a.y * s, a.y * c + a.x * s};
}

// Residues mod p (m31.cuh): both products of a component in one 64-bit sum and one fold.
__device__ __forceinline__ cpx<m31> cmul(cpx<m31> a, cpx<m31> b) {
    return {m31_fold(m31_wide(a.x, b.x) + m31_wide(a.y, -b.y)), m31_fold(m31_wide(a.x, b.y) + m31_wide(a.y, b.x))};
}
__device__ __forceinline__ cpx<m31> cmulc(cpx<m31> a, cpx<m31> b) {
    return {m31_fold(m31_wide(a.x, b.x) + m31_wide(a.y, b.y)), m31_fold(m31_wide(a.y, b.x) + m31_wide(a.x, -b.y))};
}
// x / 2
template <typename T>
__device__ __forceinline__ T halve(T x) { return T(0.5) * x; }
__device__ __forceinline__ m31 halve(m31 x) { return m31_of((x.v >> 1) | ((x.v & 1) << 30)); }

__host__ __device__ constexpr int ilog2c(int n) { return n <= 1 ? 0 : 1 + ilog2c(n >> 1); }
__host__ __device__ constexpr int brev(int k, int M) {
    int r = 0;
    for (int b = 1, t = M >> 1; b < M; b <<= 1, t >>= 1)
        if (k & b) r |= t;
    return r;
}

// cos / sin of 2*pi*k/32 from first-octant constants, so that the symmetric
// entries are exact mirror images.
__host__ __device__ constexpr double c16(int r) {
    return r == 0 ? 1.0 : r == 1 ? 0.98078528040323044913 : r == 2 ? 0.92387953251128675613
         : r == 3 ? 0.83146961230254523708 : 0.70710678118654752440;
}
__host__ __device__ constexpr double s16(int r) {
    return r == 0 ? 0.0 : r == 1 ? 0.19509032201612826785 : r == 2 ? 0.38268343236508977173
         : r == 3 ? 0.55557023301960222474 : 0.70710678118654752440;
}
__host__ __device__ constexpr double cos32q(int k) { return k <= 4 ? c16(k) : s16(8 - k); }   // k in [0, 8]
__host__ __device__ constexpr double sin32q(int k) { return k <= 4 ? s16(k) : c16(8 - k); }
__host__ __device__ constexpr double cos32(int k) {
    return k < 8 ? cos32q(k) : k < 16 ? -sin32q(k - 8) : k < 24 ? -cos32q(k - 16) : sin32q(k - 24);
}
__host__ __device__ constexpr double sin32(int k) {
    return k < 8 ? sin32q(k) : k < 16 ? cos32q(k - 8) : k < 24 ? -sin32q(k - 16) : -cos32q(k - 24);
}

// d * e^{DIR * 2 pi i k / M}, with the trivial angles special-cased.
template <int M, int DIR, typename T>
__device__ __forceinline__ cpx<T> twc(cpx<T> d, int k) {
    const int k32 = k * (32 / M);
    if (k32 == 0) return d;
    if (k32 == 8) return DIR < 0 ? cpx<T>{d.y, -d.x} : cpx<T>{-d.y, d.x};
    if (k32 == 16) return {-d.x, -d.y};
    if (k32 == 24) return DIR < 0 ? cpx<T>{-d.y, d.x} : cpx<T>{d.y, -d.x};
    return rot<DIR>(d, (T)cos32(k32), (T)sin32(k32));
}

// In-register M-point DFT, natural order in, bit-reversed order out:
// after the call v[brev(k, M)] = sum_n v_in[n] e^{DIR 2 pi i n k / M}.
// Residues: constants from the roots of unity; eighth turns are (1 +- i) 2^15, a rotation of
// the 31 bits.
template <int M, int DIR>
__device__ __forceinline__ cpx<m31> twc(cpx<m31> d, int k) {
    const int k32 = k * (32 / M);
    if (k32 == 0) return d;
    if (k32 == 8) return DIR < 0 ? cpx<m31>{d.y, -d.x} : cpx<m31>{-d.y, d.x};
    if (k32 == 16) return {-d.x, -d.y};
    if (k32 == 24) return DIR < 0 ? cpx<m31>{-d.y, d.x} : cpx<m31>{d.y, -d.x};
    if (k32 == 4 || k32 == 12) {
        auto rot15 = [](m31 a) { return m31_of(((a.v << 15) & kM31) | (a.v >> 16)); };
        const m31 s = rot15(d.x + d.y), t = rot15(d.y - d.x);  // 4: (x -+ y, y +- x); 12: i times that
        if (k32 == 4) return DIR < 0 ? cpx<m31>{s, t} : cpx<m31>{-t, s};
        return DIR < 0 ? cpx<m31>{t, -s} : cpx<m31>{-s, -t};
    }
    const uint32_t c = m31_cos32(k32), sn = m31_sin32(k32);
    return cmul(d, cpx<m31>{m31_of(c), m31_of(DIR < 0 ? kM31 - sn : sn)});
}

template <int M, int DIR, typename T>
__device__ __forceinline__ void dft_reg(cpx<T> (&v)[M]) {
#pragma unroll
    for (int span = M / 2; span >= 1; span >>= 1) {
#pragma unroll
        for (int start = 0; start < M; start += 2 * span) {
#pragma unroll
            for (int j = 0; j < span; ++j) {
                const cpx<T> a = v[start + j], b = v[start + j + span];
                v[start + j] = a + b;
                v[start + j + span] = twc<M, DIR>(a - b, j * (M / (2 * span)));
            }
        }
    }
}

}  // namespace cmif

#include "fft_pk.cuh"

namespace cmif {

// Lanes per group for a team transform: the largest power of two M with M*M
// dividing N (N = R M^2; for N = 2^k or 3 * 2^k), capped so that M complex
// values fit in registers (32 of 4-byte values, 16 of FP64).
__host__ __device__ constexpr int team_m(int N, int mmax) {
    int M = mmax;
    while (M > 1 && (M * M > N || N % (M * M) != 0)) M >>= 1;
    return M;
}
__host__ __device__ constexpr bool is_pow2(int n) { return n > 0 && (n & (n - 1)) == 0; }

// In-register R-point DFT with the output in natural order: u[q] = sum_s u_in[s]
// e^{DIR 2 pi i s q / R}.  Powers of two by the radix-2 network (the bit-reversed
// output renamed), R = 3 directly, R = 6 as two 3-point DFTs and a radix-2 step.
template <int DIR, typename T>
__device__ __forceinline__ void dft3(cpx<T>& a, cpx<T>& b, cpx<T>& c) {
    // X0 = a + b + c; X1,2 = a - (b + c)/2 -+ DIR i (sqrt(3)/2) (b - c) ... with the sign of DIR
    const T h = T(0.5), s3 = T(0.86602540378443864676);
    const cpx<T> t = {b.x + c.x, b.y + c.y}, d = {b.x - c.x, b.y - c.y};
    const cpx<T> m = {a.x - h * t.x, a.y - h * t.y};
    const cpx<T> id = {-s3 * d.y, s3 * d.x};  // i sqrt(3)/2 (b - c)
    a = {a.x + t.x, a.y + t.y};
    if (DIR > 0) {
        b = {m.x + id.x, m.y + id.y};
        c = {m.x - id.x, m.y - id.y};
    } else {
        b = {m.x - id.x, m.y - id.y};
        c = {m.x + id.x, m.y + id.y};
    }
}

template <int R, int DIR, typename T>
__device__ __forceinline__ void dft_nat(cpx<T> (&u)[R]) {
    if constexpr (R == 3) {
        dft3<DIR>(u[0], u[1], u[2]);
    } else if constexpr (R == 6) {
        // E = DFT3(u0, u2, u4), O = DFT3(u1, u3, u5); X[k] = E[k] + w6^k O[k], X[k+3] = E[k] - w6^k O[k]
        cpx<T> e0 = u[0], e1 = u[2], e2 = u[4], o0 = u[1], o1 = u[3], o2 = u[5];
        dft3<DIR>(e0, e1, e2);
        dft3<DIR>(o0, o1, o2);
        const T h = T(0.5), s3 = T(0.86602540378443864676);
        const cpx<T> w1 = {h, DIR * s3}, w2 = {-h, DIR * s3};
        o1 = cmul(o1, w1);
        o2 = cmul(o2, w2);
        u[0] = e0 + o0; u[3] = e0 - o0;
        u[1] = e1 + o1; u[4] = e1 - o1;
        u[2] = e2 + o2; u[5] = e2 - o2;
    } else {
        static_assert(is_pow2(R), "R-point DFT: powers of two, 3 and 6");
        cpx<T> t[R];
#pragma unroll
        for (int i = 0; i < R; ++i) t[i] = u[i];
        dft_reg<R, DIR>(t);
#pragma unroll
        for (int q = 0; q < R; ++q) u[q] = t[brev(q, R)];
    }
}
template <typename T>
__host__ __device__ constexpr int max_m() { return sizeof(T) == 4 ? 32 : 16; }  // 4-byte values: 32; FP64: 16

// Twiddle tables in device memory, filled once per device from FP64 values.
//   n[l][k]         = e^{-2 pi i k / 2^l},           k < 2^l
//   sq[l][k1*M + j] = e^{-2 pi i j k1 / (M*M)},       M = 2^l, j, k1 < M; FP32, M >= 8: as float4
//                     entries k*M + j, k < M/2, with rows k and k + M/2 side by side
//                     (cos, cos', sin, sin')
//   n3[l][k]        = e^{-2 pi i k / (3 2^l)},       k < 3 2^l
template <typename T>
struct Tw {
    const cpx<T>* n[14];
    const cpx<T>* sq[6];
    const cpx<T>* n3[12];
    const double2* lg;  // FP64: the c log2 c table of weighted maps (kernels.cuh)
};

// The table of e^{-2 pi i k / N} for a transform length N = 2^l or 3 2^l.
__host__ __device__ constexpr int ilog2_of(int n) { return n <= 1 ? 0 : 1 + ilog2_of(n >> 1); }
template <int N, typename T>
__device__ __forceinline__ const cpx<T>* tw_of(const Tw<T>& tw) {
    if constexpr (N % 3 == 0) return tw.n3[ilog2_of(N / 3)];
    else return tw.n[ilog2_of(N)];
}

template <int DIR, typename T>
__device__ __forceinline__ cpx<T> twl(const cpx<T>* __restrict__ t, int k) {
    cpx<T> w = t[k];
    if (DIR > 0) w.y = -w.y;
    return w;
}

// Shared-memory scratch of one group of M lanes.  Transposes of 4-byte values go through
// shared memory in two halves (real parts, then imaginary parts), so a group
// needs M*M floats; groups narrower than a warp get M floats of padding so
// that the groups of one warp hit disjoint banks.  FP64 transposes complex
// values directly.
template <int M>
__host__ __device__ constexpr int grp_pad() { return M < 32 ? M : 0; }
template <typename T, int M>
__host__ __device__ constexpr int grp_scratch_bytes() {
    return sizeof(T) == 4 ? (M * M + grp_pad<M>()) * 4 : M * M * (int)sizeof(cpx<T>);
}

// Shared memory of one team of R groups: the groups' scratch, or for R > 2 the
// N complex values of the radix-R exchange if that is more.
template <typename T, int M, int R>
__host__ __device__ constexpr int team_scratch_bytes() {
    return R > 2 && R * M * M * (int)sizeof(cpx<T>) > R * grp_scratch_bytes<T, M>()
               ? R * M * M * (int)sizeof(cpx<T>) : R * grp_scratch_bytes<T, M>();
}

// Length N = R*M*M transform by a team of R groups x M lanes.
//   load(n)  : x[n] for n in [0, N)
//   r, j     : this lane's group and lane-in-group
//   sm       : this group's scratch (grp_scratch_bytes<T, M>() bytes of shared memory);
//              for R > 2 the team's groups' scratch must start at sm - r * grp_scratch and
//              span at least N complex values (team_scratch_bytes)
//   twq      : Tw::sq for this M;  twn : Tw::n for N (used when R > 1)
// Result: v[brev(k2, M)] = X[R*(j + M*k2) + r], k2 in [0, M).
// Every lane of every warp taking part must call this (it uses __syncwarp).
// The four-step core on values already in registers: v[i] = y[j + M*i] for the
// group's M*M-point sequence y.  Result: v[brev(k2, M)] = Y[j + M*k2].
//
// FP32, M >= 8: packed DFTs (fft_pk.cuh).  The transpose holds the real and the imaginary
// parts in planes of M rows by M floats (WIDE: both planes at once, a group scratch of M*M
// complex; else one after the other).  A row's M/4 blocks of 4 floats are XOR-permuted by
// the row, so that 8 lanes reading 8 rows hit 8 different 16-byte bank groups; the writes
// of one row are a permutation of it.  Groups narrower than a warp sit in different banks
// (their padding, or WIDE: each group permutes its rows by its place in the warp).
template <int M>
__device__ __forceinline__ int tr_swz(int row) {  // the row's XOR of its block index
    return M == 32 ? row & 7 : M == 16 ? (row >> 1) & 3 : (row >> 2) & 1;
}
// Position pairs: on entry re[m] = (y[j + M 2m].re, y[j + M (2m + 1)].re); on exit re[k] =
// (Y[j + M k].re, Y[j + M (k + M/2)].re); im likewise.
template <int M, int DIR, bool WIDE>
__device__ __forceinline__ void team_core_pk(float2 (&re)[M / 2], float2 (&im)[M / 2], int j, float* sf,
                                             const float4* __restrict__ twp) {
    constexpr int H = M / 2, NB = M / 4;
    dft_pk<M, DIR>(re, im);
#pragma unroll
    for (int k = 0; k < H; ++k) {
        const float4 w = twp[k * M + j];  // rows k and k + H: (cos, cos', sin, sin'), forward sign
        const float2 c = make_float2(w.x, w.y), s = make_float2(w.z, w.w), a = re[k], b = im[k];
        if (DIR > 0) {
            re[k] = __ffma2_rn(b, s, __fmul2_rn(a, c));
            im[k] = __fmul2_rn(b, c);
            im[k] = make_float2(fmaf(-a.x, s.x, im[k].x), fmaf(-a.y, s.y, im[k].y));
        } else {
            re[k] = __fmul2_rn(a, c);
            re[k] = make_float2(fmaf(-b.x, s.x, re[k].x), fmaf(-b.y, s.y, re[k].y));
            im[k] = __ffma2_rn(a, s, __fmul2_rn(b, c));
        }
    }
    const int gx = WIDE && M < 32 ? (threadIdx.x / M) & (32 / M - 1) : 0;  // the group's place in its warp
    // byte offsets: rows sharing a block permutation x differ by whole multiples of the row
    // length, so one address per x serves all of them
    char* const base = reinterpret_cast<char*>(sf);
    auto put = [&](auto store) {
#pragma unroll
        for (int x = 0; x < NB; ++x) {
            char* const p = base + ((j << 2) ^ (x << 4));
#pragma unroll
            for (int row = 0; row < M; ++row) {
                if (tr_swz<M>(row) != x) continue;
                char* const q = WIDE && M < 32 ? p + ((row ^ gx) * M * 4) : p + row * M * 4;
                store(q, row);
            }
        }
    };
    auto get = [&](int off, float2(&d)[H]) {
        const char* const rb = base + off + (j ^ gx) * M * 4;
#pragma unroll
        for (int b = 0; b < NB; ++b) {
            const float4 q = *reinterpret_cast<const float4*>(rb + ((b ^ tr_swz<M>(j)) << 4));
            d[2 * b] = make_float2(q.x, q.y);
            d[2 * b + 1] = make_float2(q.z, q.w);
        }
    };
    auto val = [&](const float2(&d)[H], int row) { return row < H ? d[row].x : d[row - H].y; };
    __syncwarp();
    if constexpr (WIDE) {
        put([&](char* q, int row) {
            *reinterpret_cast<float*>(q) = val(re, row);
            *reinterpret_cast<float*>(q + M * M * 4) = val(im, row);
        });
        __syncwarp();
        get(0, re);
        get(M * M * 4, im);
    } else {
        put([&](char* q, int row) { *reinterpret_cast<float*>(q) = val(re, row); });
        __syncwarp();
        get(0, re);
        __syncwarp();
        put([&](char* q, int row) { *reinterpret_cast<float*>(q) = val(im, row); });
        __syncwarp();
        get(0, im);
    }
    __syncwarp();
    dft_pk<M, DIR>(re, im);
}

template <int M, int DIR, typename T>
__device__ __forceinline__ void team_fft_core(cpx<T> (&v)[M], int j, void* sm, const cpx<T>* __restrict__ twq) {
    if constexpr (std::is_same<T, float>::value && M >= 8) {
        constexpr int H = M / 2;
        float2 re[H], im[H];
#pragma unroll
        for (int m = 0; m < H; ++m) {
            re[m] = make_float2(v[2 * m].x, v[2 * m + 1].x);
            im[m] = make_float2(v[2 * m].y, v[2 * m + 1].y);
        }
        team_core_pk<M, DIR, false>(re, im, j, reinterpret_cast<float*>(sm), reinterpret_cast<const float4*>(twq));
#pragma unroll
        for (int k = 0; k < H; ++k) {
            v[brev(k, M)] = {re[k].x, im[k].x};
            v[brev(k + H, M)] = {re[k].y, im[k].y};
        }
    } else {
        auto dft = [&]() {
            if constexpr (std::is_same<T, double>::value) dft_lf<M, DIR>(v);
            else dft_reg<M, DIR>(v);
        };
        dft();  // v[brev(k1)] = A[j][k1]
#pragma unroll
        for (int k1 = 1; k1 < M; ++k1) v[brev(k1, M)] = cmul(v[brev(k1, M)], twl<DIR>(twq, k1 * M + j));
        if constexpr (sizeof(T) == 4) {
            T* sf = reinterpret_cast<T*>(sm);
            __syncwarp();
#pragma unroll
            for (int k1 = 0; k1 < M; ++k1) sf[k1 * M + (j ^ k1)] = v[brev(k1, M)].x;
            __syncwarp();
#pragma unroll
            for (int n2 = 0; n2 < M; ++n2) v[n2].x = sf[j * M + (n2 ^ j)];
            __syncwarp();
#pragma unroll
            for (int k1 = 0; k1 < M; ++k1) sf[k1 * M + (j ^ k1)] = v[brev(k1, M)].y;
            __syncwarp();
#pragma unroll
            for (int n2 = 0; n2 < M; ++n2) v[n2].y = sf[j * M + (n2 ^ j)];
            __syncwarp();
        } else {
            cpx<T>* sc = reinterpret_cast<cpx<T>*>(sm);
            __syncwarp();
#pragma unroll
            for (int k1 = 0; k1 < M; ++k1) sc[k1 * M + (j ^ k1)] = v[brev(k1, M)];
            __syncwarp();
#pragma unroll
            for (int n2 = 0; n2 < M; ++n2) v[n2] = sc[j * M + (n2 ^ j)];
            __syncwarp();
        }
        dft();  // v[brev(k2)] = X_r[j + M k2]
    }
}

// loaded(sync): called once this lane's loads are done; sync: those of the whole block are.
struct NothingOnceLoaded {
    __device__ __forceinline__ void operator()(bool) const {}
};
template <int M, int R, int DIR, typename T, typename Load, typename Loaded = NothingOnceLoaded>
__device__ __forceinline__ void team_fft(cpx<T> (&v)[M], int r, int j, Load&& load, void* sm,
                                         const cpx<T>* __restrict__ twq, const cpx<T>* __restrict__ twn,
                                         Loaded loaded = Loaded()) {
    constexpr int NQ = M * M;
    if constexpr (R > 2 && !is_pow2(R)) {
        // Radix-R decimation in frequency (R = 3, 6) with every input loaded once: the
        // team's lanes l = r M + j take the points m = l + TEAM t, form the R-point DFT
        // of x[m + s NQ], s < R, twiddle frequency q by w_N^{m q} and hand it to group q
        // through the team's buffer (as in the power-of-two case below).
        constexpr int TEAM = R * M, PTS = (NQ + TEAM - 1) / TEAM;
        cpx<T>* xs = reinterpret_cast<cpx<T>*>(reinterpret_cast<char*>(sm) - r * grp_scratch_bytes<T, M>());
        const int lt = r * M + j;
        __syncthreads();
#pragma unroll
        for (int t = 0; t < PTS; ++t) {
            const int m = lt + TEAM * t;
            if (PTS * TEAM == NQ || m < NQ) {
                cpx<T> u[R];
#pragma unroll
                for (int s2 = 0; s2 < R; ++s2) u[s2] = load(m + s2 * NQ);
                dft_nat<R, DIR>(u);
#pragma unroll
                for (int q = 0; q < R; ++q) xs[q * NQ + m] = q ? cmul(u[q], twl<DIR>(twn, m * q)) : u[q];
            }
        }
        __syncthreads();
        loaded(true);
#pragma unroll
        for (int i = 0; i < M; ++i) v[i] = xs[r * NQ + j + M * i];
        __syncthreads();
    } else if constexpr (R > 2) {
        // Radix-R decimation in frequency with every input loaded once: lane (r, j)
        // takes the points m = j + M (r PER + t), t < PER, forms the R-point DFT of
        // x[m + s NQ], s < R, in registers, twiddles frequency q by w_N^{m q} and
        // hands it to group q through the team's buffer (N complex values in front
        // of the groups' scratch: sm - r * grp_scratch).  Block-wide barriers: every
        // team of the block must call this together.
        constexpr int PER = M / R;
        static_assert(PER >= 1, "radix-R step needs R <= M");
        cpx<T>* xs = reinterpret_cast<cpx<T>*>(reinterpret_cast<char*>(sm) - r * grp_scratch_bytes<T, M>());
        __syncthreads();  // earlier users of the team's scratch are done
#pragma unroll
        for (int t = 0; t < PER; ++t) {
            const int m = j + M * (r * PER + t);
            cpx<T> u[R];
#pragma unroll
            for (int s2 = 0; s2 < R; ++s2) u[s2] = load(m + s2 * NQ);
            dft_reg<R, DIR>(u);  // u[brev(q)] = sum_s x[m + s NQ] w_R^{s q}
#pragma unroll
            for (int q = 0; q < R; ++q) {
                const cpx<T> y = u[brev(q, R)];
                xs[q * NQ + m] = q ? cmul(y, twl<DIR>(twn, m * q)) : y;
            }
        }
        __syncthreads();
        loaded(true);
#pragma unroll
        for (int i = 0; i < M; ++i) v[i] = xs[r * NQ + j + M * i];
        __syncthreads();  // the groups' transposes below reuse this buffer
    } else {
#pragma unroll
        for (int i = 0; i < M; ++i) {
            const int m = j + M * i;
            if constexpr (R == 1) {
                v[i] = load(m);
            } else {
                // radix-2 decimation in frequency: y_r[m] = w_N^{m r} (x[m] + (-1)^r x[m + NQ])
                const cpx<T> x0 = load(m), x1 = load(m + NQ);
                const cpx<T> acc = (r & 1) ? x0 - x1 : x0 + x1;
                v[i] = (r == 0) ? acc : cmul(acc, twl<DIR>(twn, m * r));
            }
        }
        loaded(false);
    }
    team_fft_core<M, DIR>(v, j, sm, twq);
}

}  // namespace cmif
