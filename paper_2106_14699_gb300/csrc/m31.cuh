// Exact transforms: complex numbers over the integers modulo the Mersenne prime
// p = 2^31 - 1.
//
// -1 is no square mod p (p = 3 mod 4), so a + b i with a, b mod p form a field of p^2
// elements, and its elements of norm a^2 + b^2 = 1 form a cyclic group of order p + 1 =
// 2^31: there are roots of unity of every order 2^k <= 2^31 whose conjugate is their inverse.
// They behave as e^{2 pi i / N} does: the transforms, the packing of two real planes per
// complex transform and the Hermitian step carry over unchanged (complex Mersenne
// transforms: Reed and Truong, IEEE Trans. Information Theory 21(2), 1975).  A correlation
// of 0/1 planes comes out as its integer count mod p; counts are at most 2^22, so they are
// exact: no rounding, no residual.  A complex product is four 32 x 32 -> 64-bit
// multiply-adds and two folds (2^31 = 1 mod p) on full-rate integer units; FP64 runs at 1/64 of
// FP32's rate on GB300, and a two-term FP32 add takes about 20 operations.  Measured, one map of
// 1024^2, K = 16: 9.1 ms (FP64 transforms 104.8, two-term FP32 79.8).
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

namespace cmif {

constexpr uint32_t kM31 = 0x7FFFFFFFu;

// A residue, 0 <= v <= p (p stands for 0 as well).
struct m31 {
    uint32_t v;
    m31() = default;
    __host__ __device__ constexpr explicit m31(int x) : v((uint32_t)x) {}
};
__host__ __device__ constexpr m31 m31_of(uint32_t v) {
    m31 r(0);
    r.v = v;
    return r;
}

__device__ __forceinline__ m31 operator+(m31 a, m31 b) {
    const uint32_t s = a.v + b.v;  // <= 2p < 2^32
    return m31_of(min(s, s - kM31));
}
__device__ __forceinline__ m31 operator-(m31 a, m31 b) {
    const uint32_t d = a.v - b.v;  // wraps when b > a; then d + p is the smaller
    return m31_of(min(d, d + kM31));
}
__device__ __forceinline__ m31 operator-(m31 a) { return m31_of(kM31 - a.v); }
// x < 2^63 (two products) modulo p: three 31-bit digits added
__device__ __forceinline__ m31 m31_fold(unsigned long long x) {
    const uint32_t t = (uint32_t)(x >> 31);
    const uint32_t s = ((uint32_t)x & kM31) + (t & kM31) + (t >> 31);  // <= 2p: t >= 2^31 leaves t & p <= p - 3
    return m31_of(min(s, s - kM31));
}
__device__ __forceinline__ unsigned long long m31_wide(m31 a, m31 b) { return (unsigned long long)a.v * b.v; }
__device__ __forceinline__ m31 operator*(m31 a, m31 b) { return m31_fold(m31_wide(a, b)); }

// The integer 0 .. 2^23 - 1 that a residue stands for, as a float.
__device__ __forceinline__ float m31_count(m31 a) {
    return __uint_as_float(0x4B000000u + (a.v == kM31 ? 0u : a.v)) - 8388608.0f;
}

// Roots of unity: u has order 2^31 and norm 1; w_N = u^(2^31 / N), w_4 = i, w_8 = 2^15 (1 + i).
struct m31c {
    uint32_t x, y;
};
__host__ __device__ constexpr uint32_t m31_mulc(uint32_t a, uint32_t b) {
    return (uint32_t)((unsigned long long)a * b % kM31);
}
__host__ __device__ constexpr m31c m31_cmul(m31c a, m31c b) {
    return {(m31_mulc(a.x, b.x) + kM31 - m31_mulc(a.y, b.y)) % kM31, (m31_mulc(a.x, b.y) + m31_mulc(a.y, b.x)) % kM31};
}
__host__ __device__ constexpr m31c m31_pow(m31c a, uint32_t n) {
    m31c r{1, 0};
    for (; n; n >>= 1) {
        if (n & 1) r = m31_cmul(r, a);
        a = m31_cmul(a, a);
    }
    return r;
}
// w_N^k, N a power of two
__host__ __device__ constexpr m31c m31_root(uint32_t k, uint32_t N) {
    return m31_pow(m31c{429496730u, 858993458u}, (uint32_t)((unsigned long long)(k % N) * (0x80000000u / N)));
}

// w_32^k = (m31_cos32(k), m31_sin32(k)): the first octant's values; w^(8 - k) = i conj(w^k)
__host__ __device__ constexpr uint32_t m31_c16(int r) {
    return r == 0 ? 1u : r == 1 ? 906276279u : r == 2 ? 1556715293u : r == 3 ? 732393395u : 32768u;
}
__host__ __device__ constexpr uint32_t m31_s16(int r) {
    return r == 0 ? 0u : r == 1 ? 967747991u : r == 2 ? 978592373u : r == 3 ? 34602070u : 32768u;
}
__host__ __device__ constexpr uint32_t m31_cq(int k) { return k <= 4 ? m31_c16(k) : m31_s16(8 - k); }
__host__ __device__ constexpr uint32_t m31_sq(int k) { return k <= 4 ? m31_s16(k) : m31_c16(8 - k); }
__host__ __device__ constexpr uint32_t m31_cos32(int k) {
    return k < 8 ? m31_cq(k) : k < 16 ? kM31 - m31_sq(k - 8) : k < 24 ? kM31 - m31_cq(k - 16) : m31_sq(k - 24);
}
__host__ __device__ constexpr uint32_t m31_sin32(int k) {
    return k < 8 ? m31_sq(k) : k < 16 ? m31_cq(k - 8) : k < 24 ? kM31 - m31_sq(k - 16) : kM31 - m31_cq(k - 24);
}

}  // namespace cmif
