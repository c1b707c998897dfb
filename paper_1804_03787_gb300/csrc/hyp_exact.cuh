// RANSAC hypotheses without double precision.
//
// GB300 runs FP64 at a small fraction of its FP32 rate, and a 4-point
// homography in FP64 was the bottleneck of the per-window fit.  Here the
// projective-basis solution H ~ B adj(A) is formed exactly in 128-bit
// integers (minimal_h_exact states their bounds) and the FP32 evaluation form is derived from exact integer numerators with one
// rounding each; the translation, which needs ~1e-7 px absolute accuracy on
// flows of hundreds of pixels, is split into hi + lo with an exact integer
// remainder.
#pragma once

#include <stdint.h>

#include "common.cuh"

namespace gpm {

typedef __int128 i128;
typedef unsigned __int128 u128;

// Integer -> float without conversion instructions (on GB300 conversions
// from 64-bit integers issue on the slow FP64 pipe): a value below 2^23 ORed
// into the mantissa of 2^23 is exact, so a 32-bit limb is two 16-bit halves
// and one fused multiply-add (correctly rounded).
__host__ __device__ __forceinline__ float u16_to_float(uint32_t v) {
#ifdef __CUDA_ARCH__
    return __int_as_float(0x4B000000u | v) - 8388608.f;
#else
    return (float)v;
#endif
}
__host__ __device__ __forceinline__ float u32_to_float(uint32_t v) {
#ifdef __CUDA_ARCH__
    return __fmaf_rn(u16_to_float(v >> 16), 65536.f, u16_to_float(v & 0xFFFFu));
#else
    return (float)v;
#endif
}

// Float near a 128-bit integer: the 32-bit limbs combined by fused multiply-adds, within about 1 ulp -- every
// caller tolerates that (the translation is corrected by an exact remainder).  Samples inside a frame stay below
// 2^92; with imported offsets far out of it mixed in, entries reach 2^111.
__host__ __device__ __forceinline__ float i128_to_float(i128 x) {
    const bool neg = x < 0;
    const u128 u = neg ? (u128)0 - (u128)x : (u128)x;  // magnitude: no cancellation between limbs
    const uint32_t l0 = (uint32_t)u, l1 = (uint32_t)(u >> 32), l2 = (uint32_t)(u >> 64), l3 = (uint32_t)(u >> 96);
#ifdef __CUDA_ARCH__
    float f = __fmaf_rn(u32_to_float(l2), 18446744073709551616.f,
                        __fmaf_rn(u32_to_float(l1), 4294967296.f, u32_to_float(l0)));
    if (l3) f = __fmaf_rn(u32_to_float(l3), 79228162514264337593543950336.f, f);
#else
    float f = (float)l2 * 18446744073709551616.f + (float)l1 * 4294967296.f + (float)l0;
    if (l3) f += (float)l3 * 79228162514264337593543950336.f;
#endif
    return neg ? -f : f;
}

// 4-point homography, exact: H = B adj(A) with the projective bases of the
// source points (A) and target points (B); window-local integer coordinates.
// With every point taken relative to the fourth pair (p3, q3), the lambdas
// are the cross products l_k of the other two source points, the target
// weights the cross products mu_k, sum_k mu_k (q_k - q3) = 0, and
//   H = T(q3) H' T(-p3),   H' = sum_k w_k (q_k - q3, 1) adj(P')_k,   w_k = mu_k l_i l_j,
// the same integers as the products with the untranslated points, in 18 wide
// products instead of 45, most of them on short factors.  For windows up to
// 96 px (|l| < 2^13.2), m the largest |mu| and q the largest target component
// or difference: |w| < 2^26.4 m, the last row < 2^42.2 m, the others < 2^43 m q.
// Targets within 2^22 (frames are below 2^15 a side): m < 2^47, |H| < 2^113;
// others (imported offsets may be any integer) only if sample_in_range.
template <class T>
__host__ __device__ inline void minimal_h_exact(const int* px, const int* py, const T* qx, const T* qy, i128* H) {
    int dx[3], dy[3];
    int64_t X[3], Y[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        dx[k] = px[k] - px[3];
        dy[k] = py[k] - py[3];
        X[k] = (int64_t)qx[k] - qx[3];
        Y[k] = (int64_t)qy[k] - qy[3];
    }
    int l[3];
    int64_t mu[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const int i = (k + 1) % 3, j = (k + 2) % 3;
        l[k] = dx[i] * dy[j] - dx[j] * dy[i];
        mu[k] = X[i] * Y[j] - X[j] * Y[i];
    }
    // H' (its third column is (0, 0, h22)); rolled: the few threads that run this wait for its instructions
    i128 h[3][2] = {}, h22 = (i128)((int64_t)l[0] * l[1] * l[2]) * (mu[0] + mu[1] + mu[2]);
#pragma unroll 1
    for (int k = 0; k < 3; ++k) {
        const int i = (k + 1) % 3, j = (k + 2) % 3;
        const i128 w = (i128)mu[k] * ((int64_t)l[i] * l[j]);
        const i128 a = w * (dy[i] - dy[j]), b = w * (dx[j] - dx[i]);
        h[0][0] += a * X[k];
        h[0][1] += b * X[k];
        h[1][0] += a * Y[k];
        h[1][1] += b * Y[k];
        h[2][0] += a;
        h[2][1] += b;
    }
    H[6] = h[2][0];
    H[7] = h[2][1];
    H[8] = h22 - h[2][0] * px[3] - h[2][1] * py[3];
    H[0] = h[0][0] + h[2][0] * qx[3];
    H[1] = h[0][1] + h[2][1] * qx[3];
    H[2] = H[8] * qx[3] - h[0][0] * px[3] - h[0][1] * py[3];
    H[3] = h[1][0] + h[2][0] * qy[3];
    H[4] = h[1][1] + h[2][1] * qy[3];
    H[5] = H[8] * qy[3] - h[1][0] * px[3] - h[1][1] * py[3];
}

// Whether minimal_h_exact and make_mef_exact hold a sample with these targets (below 2^33), moved by up to `shift`: the
// largest |mu| below 2^57 (split_ratio multiplies twice the last row by 2^24) and its product with the largest target
// below 2^82.  True of any targets within 2^22, and of targets about two places however far from each other.
__host__ __device__ inline bool sample_in_range(const int64_t* qx, const int64_t* qy, int64_t shift) {
    i128 m = 0, q = 0;
    auto raise = [](i128& a, i128 v) {
        v = v < 0 ? -v : v;
        a = v > a ? v : a;
    };
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const int i = (k + 1) % 3, j = (k + 2) % 3;
        const int64_t xi = qx[i] - qx[3], yi = qy[i] - qy[3], xj = qx[j] - qx[3], yj = qy[j] - qy[3];
        raise(m, (i128)xi * yj - (i128)xj * yi);
        raise(q, xi);
        raise(q, yi);
    }
    raise(q, qx[3]);
    raise(q, qy[3]);
    return m < (i128)1 << 57 && m * (q + shift) < (i128)1 << 82;
}

// num / den (den > 0) as hi + lo floats: hi the rounded quotient, lo the
// quotient of the exact integer remainder.
__host__ __device__ inline void split_ratio(i128 num, i128 den, float rden, float& hi, float& lo) {
    hi = i128_to_float(num) * rden;
    lo = 0.f;
    const float a = hi < 0 ? -hi : hi;
    if (!(a >= 9.5367431640625e-07f)) return;  // below 2^-20: hi alone
    int e;
#ifdef __CUDA_ARCH__
    const float mant = frexpf(hi, &e);
#else
    const float mant = __builtin_frexpf(hi, &e);
#endif
    const int sh = e < 24 ? 24 - e : 0;  // at most 44
    const i128 M = (i128)(int)(mant * 16777216.f) * ((i128)1 << (e < 24 ? 0 : e - 24));  // hi = M 2^-sh, exactly
    const i128 R = num * ((i128)1 << sh) - M * den;
#ifdef __CUDA_ARCH__
    lo = __fmul_rn(i128_to_float(R) * rden, __int_as_float((127 - sh) << 23));
#else
    lo = (i128_to_float(R) * rden) * __builtin_ldexpf(1.f, -sh);
#endif
}

// Evaluation form (origin 0) of the exact homography; false if its
// denominator vanishes at the window centre.
__host__ __device__ inline bool make_mef_exact(const i128* Hin, Mef& m) {
    i128 H[9];
    i128 dc2 = 2 * Hin[8] - (Hin[6] + Hin[7]);  // twice the denominator at the centre (-0.5, -0.5)
    if (dc2 == 0) return false;
    const bool flip = dc2 < 0;
#pragma unroll 1
    for (int k = 0; k < 9; ++k) H[k] = flip ? -Hin[k] : Hin[k];
    if (flip) dc2 = -dc2;
    const float rd = 1.f / i128_to_float(dc2);  // one reciprocal, then products (about 1 ulp each)
    float c[9];
#pragma unroll 1
    for (int k = 0; k < 9; ++k) c[k] = i128_to_float(2 * H[k] - ((k & 3) == 0 ? dc2 : 0)) * rd;  // k = 0, 4, 8: less 1
    m.b0 = c[0];
    m.h1 = c[1];
    m.h3 = c[3];
    m.b4 = c[4];
    m.g0 = c[6];
    m.g1 = c[7];
    m.e0 = c[8];
    float t[2][2];
#pragma unroll 1
    for (int k = 0; k < 2; ++k) split_ratio(2 * H[2 + 3 * k], dc2, rd, t[k][0], t[k][1]);
    m.h2h = t[0][0];
    m.h2l = t[0][1];
    m.h5h = t[1][0];
    m.h5l = t[1][1];
    m.ef = 0.f;
    m.ox = 0;
    m.oy = 0;
    m.valid = 0;
    m.eden = 0;
    return true;
}

// Bit length of a 128-bit magnitude (0 for zero).
__host__ __device__ __forceinline__ int u128_bits(u128 u) {
    const uint64_t hi = (uint64_t)(u >> 64), lo = (uint64_t)u;
#ifdef __CUDA_ARCH__
    return hi ? 128 - __clzll((long long)hi) : (lo ? 64 - __clzll((long long)lo) : 0);
#else
    return hi ? 128 - __builtin_clzll(hi) : (lo ? 64 - __builtin_clzll(lo) : 0);
#endif
}

// The 9 entries of an exact homography as doubles scaled by one power of two
// (the largest magnitude in [1, 2)), each truncated to 53 significant bits,
// with every sign flipped when flip is set.  Built from integer operations
// alone: the exponent and mantissa fields are assembled directly (on GB300 a
// 64-bit integer conversion or an FP64 divide issues on the slow FP64 pipe).
__host__ __device__ inline void exact_to_double_pow2(const i128* H, double* D, bool flip) {
    int bl[9], E = 0;
#pragma unroll 1
    for (int k = 0; k < 9; ++k) {
        const u128 u = H[k] < 0 ? (u128)0 - (u128)H[k] : (u128)H[k];
        bl[k] = u128_bits(u);
        E = bl[k] > E ? bl[k] : E;
    }
#pragma unroll 1
    for (int k = 0; k < 9; ++k) {
        const bool neg = H[k] < 0;
        const u128 u = neg ? (u128)0 - (u128)H[k] : (u128)H[k];
        uint64_t bits = 0;
        if (bl[k] > 0) {
            // m: the leading 53 bits, value m 2^(bl - 53); scaled by 2^-E: m 2^(bl - E - 53), whose biased
            // exponent field is bl - E + 1022 + 1 (>= 897 for magnitudes below 2^127: always normal)
            const uint64_t m = bl[k] > 53 ? (uint64_t)(u >> (bl[k] - 53)) : (uint64_t)u << (53 - bl[k]);
            bits = ((uint64_t)(bl[k] - E + 1023) << 52) | (m & 0xFFFFFFFFFFFFFull);
            if (neg != flip) bits |= 0x8000000000000000ull;
        }
#ifdef __CUDA_ARCH__
        D[k] = __longlong_as_double((long long)bits);
#else
        __builtin_memcpy(&D[k], &bits, 8);
#endif
    }
}

// The first n entries of an exact homography as doubles (unnormalised).
__host__ __device__ inline void exact_to_double(const i128* H, double* D, int n = 9) {
#pragma unroll 1
    for (int k = 0; k < n; ++k) {
        const bool neg = H[k] < 0;
        const u128 u = neg ? (u128)0 - (u128)H[k] : (u128)H[k];
        const double v = (double)(uint64_t)(u >> 64) * 18446744073709551616.0 + (double)(uint64_t)u;
        D[k] = neg ? -v : v;
    }
}

}  // namespace gpm
