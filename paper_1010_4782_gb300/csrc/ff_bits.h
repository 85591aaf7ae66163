// ff_bits.h - FP64 <-> float-float pairs by integer arithmetic on the numbers' bits.
//
// The conversions between FP64 and FP32 and the FP64 additions that these replace run on
// GB300's FP64 pipe at two lanes per cycle and SM, which bound the vector conversions
// (32^3 x 64: pack and unpack run in 19 and 20 us, 100 MB each).  The results are the same
// bits.  Compiles for the host too, where the tests compare every edge with it.
#pragma once

#include <cstring>

#if defined(__CUDACC__)
#include <cuda_runtime.h>
#define STAG_BITS_FN __host__ __device__ __forceinline__
#else
#define STAG_BITS_FN inline
#endif

namespace stag {

struct FFPair {
    float hi, lo;
};

template <class To, class From>
STAG_BITS_FN To bits_as(From v) {
    static_assert(sizeof(To) == sizeof(From), "same size");
    To t;
    memcpy(&t, &v, sizeof(t));
    return t;
}

// hi = fl32(a), lo = fl32(a - hi), for exponents from 2^-70 to 2^120 by integer arithmetic.
STAG_BITS_FN FFPair ff_split(double a) {
    const unsigned long long b = bits_as<unsigned long long>(a);
    const unsigned int h = (unsigned int)(b >> 32), l = (unsigned int)b;
    const int e = (int)((h >> 20) & 0x7ffu) - 1023;
    if (e < -70 || e > 120) {  // zero, tiny, huge, not finite
        const float hi = (float)a;
        return FFPair{hi, (float)(a - (double)hi)};
    }
    // significand: 24 bits q and 29 bits below them, rounded to nearest even
    unsigned int q = ((h & 0xfffffu) << 3) | 0x800000u | (l >> 29);
    int rem = (int)(l & 0x1fffffffu);
    const bool up = rem > 0x10000000 || (rem == 0x10000000 && (q & 1u));
    if (up) {
        q += 1;
        rem -= 0x20000000;
    }
    const unsigned int sign = h & 0x80000000u;
    if (sign) rem = -rem;
    const float hi = bits_as<float>(sign | (((unsigned int)(e + 127) << 23) + (q - 0x800000u)));
    const float lo = (float)rem * bits_as<float>((unsigned int)(e - 52 + 127) << 23);
    return FFPair{hi, lo};
}

// (double)hi + (double)lo, rounded to nearest even; by integer arithmetic where hi is a normal
// number of ordinary size and lo less than a unit in its last place (TwoSum leaves at most
// half of one); a larger lo could carry past the bit that the rounding expects to lead.
STAG_BITS_FN double ff_sum(float hi, float lo) {
    const unsigned int h = bits_as<unsigned int>(hi), l = bits_as<unsigned int>(lo);
    const int eh = (int)((h >> 23) & 0xff), el = (int)((l >> 23) & 0xff);
    const bool lo_zero = (l << 1) == 0u;
    if (eh < 40 || eh > 250 || !(lo_zero || (el >= 1 && eh - el >= 24))) return (double)hi + (double)lo;
    // 24-bit significands; hi's leading bit at 61, lo's bits below the shift kept as a sticky one
    unsigned long long s = (unsigned long long)((h & 0x7fffffu) | 0x800000u) << 38;
    if (!lo_zero) {
        const unsigned long long m = (l & 0x7fffffu) | 0x800000u;
        const int shift = 38 - (eh - el);
        unsigned long long t;
        if (shift >= 0)
            t = m << shift;
        else if (shift > -24)
            t = (m >> -shift) | ((m & ((1ull << -shift) - 1ull)) != 0ull);
        else
            t = 1ull;
        s = ((h ^ l) & 0x80000000u) ? s - t : s + t;
    }
    int e = eh - 127;
    if (!(s >> 61)) {
        s <<= 1;
        e -= 1;
    }
    unsigned long long q = s >> 9;
    const unsigned int rem = (unsigned int)s & 0x1ffu;
    q += rem > 0x100u || (rem == 0x100u && (q & 1ull));
    const unsigned long long bits = ((unsigned long long)(h & 0x80000000u) << 32) |
                                    (((unsigned long long)(e + 1023) << 52) + (q - (1ull << 52)));
    return bits_as<double>(bits);
}

// ---- sums of FP32 numbers in 64-bit fixed point
// The unit is 2^-56 of 2^(E - 127), E the largest biased exponent of the numbers added: a
// number is below 2^57 units and exact unless it is more than 2^33 times smaller than
// the largest.
STAG_BITS_FN int float_exponent(float x) {  // biased; 1 for zero and subnormals
    const int e = (int)((bits_as<unsigned int>(x) >> 23) & 0xffu);
    return e ? e : 1;
}

// x in units, rounded to nearest (E >= float_exponent(x), x finite).
STAG_BITS_FN long long float_to_fixed(float x, int E) {
    const unsigned int b = bits_as<unsigned int>(x);
    const unsigned int m = (b & 0x7fffffu) | ((b & 0x7f800000u) ? 0x800000u : 0u);
    const int shift = 33 - (E - float_exponent(x));
    long long v = 0;
    if (shift >= 0)
        v = (long long)((unsigned long long)m << shift);
    else if (shift >= -24)
        v = (long long)((m + (1u << (-shift - 1))) >> -shift);
    return (b >> 31) ? -v : v;
}

// v units in FP64, rounded to nearest even.
STAG_BITS_FN double fixed_to_double(long long v, int E) {
    if (v == 0) return 0.0;
    const unsigned long long sign = (unsigned long long)v & 0x8000000000000000ull;
    const unsigned long long u = sign ? 0ull - (unsigned long long)v : (unsigned long long)v;
#if defined(__CUDA_ARCH__)
    const int lz = __clzll((long long)u);
#else
    const int lz = __builtin_clzll(u);
#endif
    const unsigned long long n = u << lz;  // leading bit at 63
    unsigned long long q = n >> 11;
    const unsigned int rem = (unsigned int)n & 0x7ffu;
    q += rem > 0x400u || (rem == 0x400u && (q & 1ull));
    const int e = 63 - lz + E - (127 + 56);
    return bits_as<double>(sign | (((unsigned long long)(e + 1023) << 52) + (q - (1ull << 52))));
}

}  // namespace stag
