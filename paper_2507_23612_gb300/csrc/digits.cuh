// Digit form of real numbers for exact products on the FP16 tensor cores (the splitting of
// Ozaki, Ogita, Oishi and Rump, Numer. Algorithms 59 (2012), with FP16 operands and FP32
// accumulation as in Mukunoki, Ozaki, Ogita and Imamura, ISC 2020).
//
// Numbers that share a scale (a column, a function) become integers relative to the largest
// magnitude of the group, of 54 bits (double) or 30 bits (float), written as S = 7 or 4
// signed base-256 digits d_1 .. d_S in [-128, 127] (|d_1| <= 64).  FP16 holds every digit
// exactly, a product of two digits is an integer of at most 14 bits and the FP32 accumulator
// of the tensor core holds integers up to 2^24.  A level l = i + j - 1 (digits i and j) has l
// products, of at most (l - 2) 2^14 + 2 x 2^13 together (2^12 for l = 1):
//
//   terms    sums within 2^24 whatever the digits
//   256      levels 1 - 5 (6 and 7 can pass it by a quarter and a half)
//   512      levels 1 - 3
//
// and an accumulator beyond 2^24 drops the odd unit of an addition.  The double forms (S = 7) sum at
// most 256 terms: what levels 6 and 7 can lose is under 2^-54 of a sum of products that are all
// that large.  With 512 it would be 2^-40 (level 4).  The float forms (S = 4, in Gram products
// and rotations 5 levels) sum up to 512, with at most 2^-37.  Levels beyond are dropped (2^-56 and
// 2^-32 of the largest product; 2^-40 with 5 levels).
//
// The bits are relative to the largest magnitude of the group: a number 2^-k of it has k bits
// fewer, down to none, where a floating-point operand would keep all of its own.  So groups are
// small where the results are local: the values of X around a brick (gather), the coefficients of a
// brick's functions (scatter), the orbitals at a point (rotation); a Gram product, which is a norm, takes
// whole columns.
#pragma once
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <cstdint>

namespace hub {

template <typename R> struct Digits;
template <> struct Digits<double> {
    static constexpr int S = 7;
    static constexpr int kEmin = 123, kEmax = 1923;        // biased exponents covered
    static constexpr int kUnit = 1076;                     // value = integer * 2^(E - kUnit)
    static constexpr int kBias = 1023;
    using I = unsigned long long;
    static constexpr I kZero = 0x80808080808080ull;
    static __device__ __forceinline__ int exponent(double v) { return (__double2hiint(v) >> 20) & 0x7ff; }
    // integer with the digits as its bytes (offset by 128 each), for a value of biased exponent
    // e = exponent(v) + de in a group whose largest is E (E >= e, E >= kEmin).  With de = 0 a zero or
    // denormal v shifts to zero whatever its hidden bit; with another de the caller leaves it out
    static __device__ __forceinline__ I bytes(double v, int E, int de = 0) {
        const unsigned hi = (unsigned)__double2hiint(v), lo = (unsigned)__double2loint(v);
        const int sh = min(E - de - ((int)(hi >> 20) & 0x7ff), 63);
        const I t = (((I)((hi & 0xfffffu) | 0x100000u) << 32 | lo) << 2) >> sh;
        // t / 2 to nearest, the offset added before the shift; a negative one through ~t, so that
        // halves go away from zero for both signs (no bias)
        return ((t ^ (I)(long long)((int)hi >> 31)) + 0x101010101010101ull) >> 1;
    }
};
template <> struct Digits<float> {
    static constexpr int S = 4;
    static constexpr int kEmin = 40, kEmax = 214;
    static constexpr int kUnit = 156;
    static constexpr int kBias = 127;
    using I = unsigned;
    static constexpr I kZero = 0x80808080u;
    static __device__ __forceinline__ int exponent(float v) { return (__float_as_int(v) >> 23) & 0xff; }
    static __device__ __forceinline__ I bytes(float v, int E, int de = 0) {
        const unsigned u = __float_as_uint(v);
        const int sh = min(E - de - ((int)(u >> 23) & 0xff), 31);
        const unsigned t = (((u & 0x7fffffu) | 0x800000u) << 7) >> sh;
        return (unsigned)(((int)(t ^ (unsigned)((int)u >> 31)) + 1) >> 1) + 0x80808080u;
    }
};

// digit j (0: most significant) of two numbers as a half2
template <typename R>
__device__ __forceinline__ __half2 digit_pair(typename Digits<R>::I a, typename Digits<R>::I b, int j) {
    const int byte = Digits<R>::S - 1 - j;
    unsigned wa, wb;
    if constexpr (sizeof(R) == 8) {
        wa = byte >= 4 ? (unsigned)(a >> 32) : (unsigned)a;
        wb = byte >= 4 ? (unsigned)(b >> 32) : (unsigned)b;
    } else {
        wa = a;
        wb = b;
    }
    const unsigned q = byte & 3;
    // bytes [a, -, b, -]; 0x6400 | b is the FP16 number 1024 + b
    unsigned t = __byte_perm(wa, wb, q | (q << 4) | ((4 + q) << 8) | ((4 + q) << 12));
    t = (t & 0x00ff00ffu) | 0x64006400u;
    return __hsub2(*reinterpret_cast<__half2*>(&t), __half2half2(__ushort_as_half(0x6480)));   // - 1152
}

// x * 2^k: an integer addition where x and the result are normal
__device__ __forceinline__ double scale2(double x, int k) {
    const int hi = __double2hiint(x), e = (hi >> 20) & 0x7ff;
    if (e == 0 || (unsigned)(e + k - 1) >= 2046u) return scalbn(x, k);
    return __hiloint2double(hi + (k << 20), __double2loint(x));
}

// the S level sums of one product (exact integers in FP32) as a double times 2^-shift:
// sum_l v[l] 256^(S - 1 - l) = result * 2^shift
template <typename R, int STRIDE>
__device__ __forceinline__ long long level_sum(const uint32_t* v, long long* low) {
    long long z[Digits<R>::S];
#pragma unroll
    for (int l = 0; l < Digits<R>::S; ++l) z[l] = __float2int_rn(__uint_as_float(v[l * STRIDE]));
    const long long hi = ((z[0] << 24) + (z[1] << 16)) + ((z[2] << 8) + z[3]);
    if constexpr (sizeof(R) == 8) *low = ((z[4] << 16) + (z[5] << 8)) + z[6];
    else *low = 0;
    return hi;
}

}  // namespace hub
