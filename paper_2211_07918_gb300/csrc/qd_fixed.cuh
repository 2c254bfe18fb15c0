// Sums of products in FP64 quality on the integer units.
//
// The FP64 pipe of this chip issues two lanes per SM and clock (1.25 TFLOP/s
// over the GPU), and conversions from FP32 go through it too: a readout that
// widens both parts of an amplitude and squares them in FP64 takes five such
// operations per amplitude, 8 ps against the 1.2 ps that reading the
// amplitude takes at the copy rate.  The integer units have 32-64 times that
// rate, and the products involved are exact integers: the mantissas of two
// complex64 parts multiply to 48 bits.  The routines below take a small group
// of products, align them to the group's largest exponent in 64-bit integers
// (one truncation of at most 2^-57 of the group's largest product each), add
// them exactly and return the group's sum as one correctly rounded double:
// one FP64 operation per group remains (adding it to the caller's sum).
//
// Groups that the alignment does not cover (infinities, NaN, only denormal or
// extremely small or large parts) take the plain FP64 expression.
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

#include "qd_common.cuh"

namespace qd {

// Right shift that is 0 from 64 on (the PTX shift clamps).
__device__ __forceinline__ uint64_t shr64(uint64_t v, uint32_t s) {
    uint64_t r;
    asm("shr.b64 %0, %1, %2;" : "=l"(r) : "l"(v), "r"(s));
    return r;
}

// v * 2^e for an unsigned integer v, round to nearest even; the result must
// be a normal double (callers bound e).
__device__ __forceinline__ double u64_scaled(uint64_t v, int e) {
    if (v == 0) return 0.0;
    const int z = __clzll((long long)v);
    v <<= z;                                   // top bit at 63: v = m 2^-z
    uint64_t m = v >> 11;                      // 53 bits, the implicit one at bit 52
    const uint32_t rest = (uint32_t)v & 0x7ffu;
    // half up, ties to even; a carry out of the mantissa moves the exponent by itself
    m += (rest > 0x400u || (rest == 0x400u && (m & 1u))) ? 1u : 0u;
    return __longlong_as_double((long long)(m + ((uint64_t)(uint32_t)(e + 63 - z + 1022) << 52)));
}

__device__ __forceinline__ double s64_scaled(int64_t v, int e) {
    const double r = u64_scaled((uint64_t)(v < 0 ? -v : v), e);
    return v < 0 ? -r : r;
}

// A part of an amplitude as an integer: value = (hi 2^32 + lo) 2^(ex - 1086),
// hi's top bit set, or hi = lo = 0.  lo is 0 for an FP32 part (and constant,
// so that its products fold away).
struct Mant {
    uint32_t hi, lo, sign;  // sign: 0 or ~0
    int ex;                 // FP64-biased exponent
};
__device__ __forceinline__ Mant mant_of(float x) {
    const uint32_t b = __float_as_uint(x), u = b & 0x7fffffffu;
    return Mant{u ? (b << 8) | 0x80000000u : 0u, 0u, (uint32_t)((int32_t)b >> 31), (int)(u >> 23) + 896};
}
__device__ __forceinline__ Mant mant_of(double x) {
    const uint32_t h = (uint32_t)__double2hiint(x), l = (uint32_t)__double2loint(x);
    const bool nz = ((h & 0x7fffffffu) | l) != 0u;
    return Mant{nz ? (h << 11) | (l >> 21) | 0x80000000u : 0u, l << 11, (uint32_t)((int32_t)h >> 31),
                (int)((h >> 20) & 0x7ffu)};
}
// The leading word of a part without its sign: orders parts by magnitude.
__device__ __forceinline__ uint32_t abs_bits(float x) { return __float_as_uint(x) & 0x7fffffffu; }
__device__ __forceinline__ uint32_t abs_bits(double x) { return (uint32_t)__double2hiint(x) & 0x7fffffffu; }
// Exponent of the larger part of an amplitude, in the FP64 bias.
__device__ __forceinline__ int amp_ex(const float2 a) {
    return (int)(max(abs_bits(a.x), abs_bits(a.y)) >> 23) + 896;
}
__device__ __forceinline__ int amp_ex(const double2 a) {
    return (int)(max(abs_bits(a.x), abs_bits(a.y)) >> 20);
}
// amp_ex of an infinity or NaN.
template <typename T> constexpr int kExInf = sizeof(T) == 4 ? 255 + 896 : 2047;

// Leading 64 bits of the product of two mantissas, in [2^62, 2^64) (below by
// at most 3 units), or 0.
__device__ __forceinline__ uint64_t mant_mul(const Mant &a, const Mant &b) {
    uint64_t p = (uint64_t)a.hi * b.hi;
    if (a.lo) p += ((uint64_t)a.lo * b.hi) >> 32;
    if (b.lo) p += ((uint64_t)a.hi * b.lo) >> 32;
    return p;
}

template <typename T>
__device__ __forceinline__ double prob64(const v2<T> a) {
    const double x = (double)a.x, y = (double)a.y;
    return fma(x, x, y * y);
}

// Range of a group's largest exponent (FP64 bias) in which the aligned sum
// applies: below it a denormal part (read here as if it had its implicit bit)
// would not be aligned away entirely; above it a sum could leave the doubles.
template <typename T> constexpr int kExLow = sizeof(T) == 4 ? 960 : 700;
template <typename T> constexpr int kExTop = sizeof(T) == 4 ? kExInf<float> : 1500;

// Sum of |v_i|^2 over a group of G amplitudes (2 G squares below 2^(64 - S)).
// The ALU pipe bounds it (64 lanes per SM and clock; 9 of its operations per
// part): the largest part is found on the raw bits, and a zero needs no test
// (its exponent field shifts it out).
template <typename T, int G>
__device__ __forceinline__ double group_norm(const v2<T> *v) {
    static_assert(G == 1 || G == 2 || G == 4 || G == 8, "group size");
    constexpr uint32_t S = G == 1 ? 1 : G == 2 ? 2 : G == 4 ? 3 : 4;
    uint32_t top = 0;
#pragma unroll
    for (int i = 0; i < G; ++i) top = max(top, max(abs_bits(v[i].x), abs_bits(v[i].y)));
    const int E = sizeof(T) == 4 ? (int)(top >> 23) + 896 : (int)(top >> 20);
    if (E >= kExLow<T> && E < kExTop<T>) {
        uint64_t acc = 0;
#pragma unroll
        for (int i = 0; i < 2 * G; ++i) {
            const T c = i & 1 ? v[i / 2].y : v[i / 2].x;
            if constexpr (sizeof(T) == 4) {
                const uint32_t u = abs_bits(c), m = (u << 8) | 0x80000000u;
                acc += shr64((uint64_t)m * m, (S + 2u * (top >> 23)) - 2u * (u >> 23));
            } else {
                const Mant x = mant_of(c);
                // hi^2 + 2 hi lo: the square's leading 64 bits
                const uint64_t p = (uint64_t)x.hi * x.hi + (((uint64_t)x.hi * x.lo) >> 31);
                acc += shr64(p, S + 2u * (uint32_t)(E - x.ex));
            }
        }
        return u64_scaled(acc, 2 * E - 2108 + (int)S);
    }
    double s = 0.0;
    if (top)
#pragma unroll
        for (int i = 0; i < G; ++i) s += prob64<T>(v[i]);
    return s;
}

// re, im of the sum of conj(a_i) b_i over a group of G amplitudes.  Aligned
// to the largest |a_i| |b_i| of the group, so that an amplitude that is large
// in one state and small in the other costs no accuracy.
template <typename TA, typename TB, int G>
__device__ __forceinline__ void group_overlap(const v2<TA> *a, const v2<TB> *b, double &re, double &im) {
    constexpr uint32_t S = G <= 2 ? 3 : 4;  // 2 G signed terms below 2^63
    static_assert(G <= 4, "group size");
    int E = 0, top = 0, topb = 0;
#pragma unroll
    for (int i = 0; i < G; ++i) {
        const int ea = amp_ex(a[i]), eb = amp_ex(b[i]);
        top = max(top, ea);
        topb = max(topb, eb);
        E = max(E, ea + eb);
    }
    // the largest product at least 2^-46, amplitudes below 2^10: a denormal part is aligned away
    if (E >= 2000 && top < 1033 && topb < 1033) {
        int64_t sr = 0, si = 0;
#pragma unroll
        for (int i = 0; i < G; ++i) {
            const Mant ax = mant_of(a[i].x), ay = mant_of(a[i].y), bx = mant_of(b[i].x), by = mant_of(b[i].y);
            auto term = [&](const Mant &p, const Mant &q, uint32_t flip) {
                const int64_t t = (int64_t)shr64(mant_mul(p, q), S + (uint32_t)(E - p.ex - q.ex));
                const int64_t sg = (int64_t)(int32_t)(p.sign ^ q.sign ^ flip);
                return (t ^ sg) - sg;
            };
            sr += term(ax, bx, 0u) + term(ay, by, 0u);
            si += term(ax, by, 0u) + term(ay, bx, ~0u);
        }
        re = s64_scaled(sr, E - 2108 + (int)S);
        im = s64_scaled(si, E - 2108 + (int)S);
        return;
    }
    re = im = 0.0;
#pragma unroll
    for (int i = 0; i < G; ++i) {
        const double xr = (double)a[i].x, xi = (double)a[i].y, yr = (double)b[i].x, yi = (double)b[i].y;
        re = fma(xr, yr, fma(xi, yi, re));
        im = fma(xr, yi, fma(-xi, yr, im));
    }
}

// |a|^2 of one amplitude, rounded once (as fma(x, x, y * y) of the exact
// squares): complex64 squares are 48-bit integers, placed into doubles by
// shifts, and one FP64 addition remains.
__device__ __forceinline__ double square_f32(float x) {
    const uint32_t u = __float_as_uint(x) & 0x7fffffffu;
    const uint32_t m = (u & 0x7fffffu) | 0x800000u;
    const uint64_t p = (uint64_t)m * m;               // in [2^46, 2^48)
    const uint32_t t = (uint32_t)(p >> 47);           // 1 from 2^47 on
    const uint64_t bits = (p << (6u - t)) + ((uint64_t)(((u >> 22) & 0x1feu) + 768u + t) << 52);
    return __longlong_as_double((long long)(u ? bits : 0ull));
}
__device__ __forceinline__ bool ordinary(float x) {  // zero or a normal number
    const uint32_t u = __float_as_uint(x) & 0x7fffffffu;
    return u == 0u || (u - 0x800000u) < 0x7f000000u;
}
__device__ __forceinline__ double prob_of(const float2 a) {
    if (ordinary(a.x) && ordinary(a.y)) return square_f32(a.x) + square_f32(a.y);
    return prob64<float>(a);
}
__device__ __forceinline__ double prob_of(const double2 a) { return prob64<double>(a); }

}  // namespace qd
