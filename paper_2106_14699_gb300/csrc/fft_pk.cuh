// Packed FP32 DFTs: two values side by side in every register pair.
//
// The register DFTs of the team transforms are issue-bound: a scalar radix-2
// network of 32 points issues 388 to 432 instructions.  sm_100+ has two-lane FP32
// instructions (FADD2 / FFMA2), which do two equal operations in one issue slot,
// so the M-point DFT is split by decimation in time into the DFTs of its even and
// odd inputs, and these two run side by side in the two lanes (same constants,
// same steps; multiplying by +-i only renames registers).  The last stage joins
// the lanes with scalar butterflies.  32 points: 148 packed + 92 scalar
// instructions.
//
// A butterfly e +- w o with w = cos + i sin takes six operations instead of eight:
// with t = tan (or cot, whichever is at most 1 in magnitude) u = o.re - t o.im,
// v = o.im + t o.re, then e +- cos (u + i v), each one fused multiply-add (the
// factored-rotation form of Linzer and Feig, IEEE Trans. Signal Processing 41(1),
// 1993).  It rounds less often than product-then-sum.
#pragma once
#include <cuda_runtime.h>

namespace cmif {

// FP64 register DFTs (weighted maps) take the same butterflies: 16 points in 148 instead of 168
// FP64 instructions, which run at 1/64 rate.

// a * k + b and a - b for scalars and for pairs (k a compile-time constant)
__device__ __forceinline__ double fmak(double a, double k, double b) { return fma(a, k, b); }
__device__ __forceinline__ double addv(double a, double b) { return a + b; }
__device__ __forceinline__ double subv(double a, double b) { return a - b; }
__device__ __forceinline__ float fmak(float a, float k, float b) { return fmaf(a, k, b); }
__device__ __forceinline__ float2 fmak(float2 a, float k, float2 b) { return __ffma2_rn(a, make_float2(k, k), b); }
__device__ __forceinline__ float addv(float a, float b) { return a + b; }
__device__ __forceinline__ float2 addv(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float subv(float a, float b) { return a - b; }
__device__ __forceinline__ float2 subv(float2 a, float2 b) { return __ffma2_rn(b, make_float2(-1.f, -1.f), a); }

// (e, o) <- (e + w o, e - w o), w = e^{DIR 2 pi i k / 32}, 0 <= k < 16
template <int DIR, typename V>
__device__ __forceinline__ void bfly(V& er, V& ei, V& orr, V& oi, int k) {
    if (k == 0) {
        const V a = er, b = ei;
        er = addv(a, orr);
        ei = addv(b, oi);
        orr = subv(a, orr);
        oi = subv(b, oi);
    } else if (k == 8) {  // w = DIR i
        const V a = er, b = ei, x = orr, y = oi;
        if (DIR > 0) {
            er = subv(a, y);
            ei = addv(b, x);
            orr = addv(a, y);
            oi = subv(b, x);
        } else {
            er = addv(a, y);
            ei = subv(b, x);
            orr = subv(a, y);
            oi = addv(b, x);
        }
    } else {
        using K = typename std::conditional<std::is_same<V, double>::value, double, float>::type;
        const double c = cos32(k), s = DIR > 0 ? sin32(k) : -sin32(k);
        const V a = er, b = ei;
        if (c * c >= s * s) {
            const K t = (K)(s / c), cf = (K)c;
            const V u = fmak(oi, -t, orr), v = fmak(orr, t, oi);
            er = fmak(u, cf, a);
            ei = fmak(v, cf, b);
            orr = fmak(u, -cf, a);
            oi = fmak(v, -cf, b);
        } else {
            const K t = (K)(c / s), sf = (K)s;
            const V u = fmak(orr, -t, oi), v = fmak(oi, t, orr);
            er = fmak(u, -sf, a);
            ei = fmak(v, sf, b);
            orr = fmak(u, sf, a);
            oi = fmak(v, -sf, b);
        }
    }
}

// M-point DFT of x, held as pairs re[m] = (x[2m].re, x[2m + 1].re) (im likewise).
// Afterwards re[k] = (X[k].re, X[k + M/2].re): natural order.
template <int M, int DIR>
__device__ __forceinline__ void dft_pk(float2 (&re)[M / 2], float2 (&im)[M / 2]) {
    constexpr int H = M / 2;
    float2 a[H], b[H];
#pragma unroll
    for (int i = 0; i < H; ++i) {
        a[i] = re[brev(i, H)];
        b[i] = im[brev(i, H)];
    }
#pragma unroll
    for (int half = 1; half < H; half <<= 1)
#pragma unroll
        for (int s = 0; s < H; s += 2 * half)
#pragma unroll
            for (int k = 0; k < half; ++k)
                bfly<DIR>(a[s + k], b[s + k], a[s + k + half], b[s + k + half], k * (16 / half));
#pragma unroll
    for (int k = 0; k < H; ++k) {
        bfly<DIR>(a[k].x, b[k].x, a[k].y, b[k].y, k * (16 / H));
        re[k] = a[k];
        im[k] = b[k];
    }
}

// The same network on scalars: M-point DFT of v, natural order in, bit-reversed order out
// (v[brev(k, M)] = X[k], as dft_reg).
template <int M, int DIR, typename T>
__device__ __forceinline__ void dft_lf(cpx<T> (&v)[M]) {
    T a[M], b[M];
#pragma unroll
    for (int i = 0; i < M; ++i) {
        a[i] = v[brev(i, M)].x;
        b[i] = v[brev(i, M)].y;
    }
#pragma unroll
    for (int half = 1; half < M; half <<= 1)
#pragma unroll
        for (int s = 0; s < M; s += 2 * half)
#pragma unroll
            for (int k = 0; k < half; ++k)
                bfly<DIR>(a[s + k], b[s + k], a[s + k + half], b[s + k + half], k * (16 / half));
#pragma unroll
    for (int k = 0; k < M; ++k) v[brev(k, M)] = {a[k], b[k]};
}

}  // namespace cmif
