// Unpacking of fp64 packed results (eqs. 9-10 and 13-14) in integer arithmetic.
//
// GB300 runs every fp64 operation -- add, multiply, fma, rint and the
// conversions to and from integers alike -- at 2 lanes per clock and SM
// (measured: 1.8-2.2), against 64-128 for integer instructions.  The packed
// main loop keeps that pipe full, so each fp64 operation the unpack spends per
// output and slab costs as much as a packed multiply-accumulate: rint, scale,
// rint and fma were 4 of the 48 (W = 3) or 69 (W = 2) fp64 operations per
// output and slab at L = 128.  The digits are therefore taken from the bits of
// the packed result on the integer pipes; only the fma into the running sum is
// left on the fp64 pipe.
//
// Every function returns the double that the fp64 form of the equations gives
// (a zero digit may differ in its sign, which no running sum carries: they
// start at +0 and only add).
#pragma once

#include <stdint.h>

namespace tdg {

// The fp64 value of an integer of at most 53 significant bits.
__device__ inline double double_of_bits(long long v) {
    const unsigned long long a = v < 0 ? 0ull - (unsigned long long)v : (unsigned long long)v;
    const int lz = __clzll((long long)a);          // 64 for a = 0
    unsigned long long b = ((unsigned long long)(1085 - lz) << 52) + ((a << (lz & 63)) >> 11);
    b = a ? b : 0ull;
    return __longlong_as_double((long long)(b | ((unsigned long long)v & 0x8000000000000000ull)));
}
__device__ inline double double_of_bits(int v) {
    const unsigned int a = v < 0 ? 0u - (unsigned int)v : (unsigned int)v;
    const int lz = __clz((int)a);                  // 32 for a = 0
    const unsigned int m = a << (lz & 31);
    const int hi = (int)(((unsigned int)(1053 - lz) << 20) + (m >> 11));
    return __hiloint2double((a ? hi : 0) | (v & (int)0x80000000), (int)(m << 21));
}

// Round to nearest, ties to even, of f 2^-s, |f| < 2^53, s >= 1.  (From s = 54
// on the value lies below one half, and the clamped shift gives 0.)
__device__ inline long long rne_shift(long long f, int s) {
    s = s < 54 ? s : 54;
    return (f + ((1ll << (s - 1)) - 1) + ((f >> s) & 1)) >> s;
}

// Symmetric form: u = rint(r), t = rint(z u), u - Q t with Q = 2^q: the low q
// bits of u as a signed number.  When they are exactly half of Q, t is a tie
// that goes to the even integer: +Q/2 if bit q of u (the parity of floor(u/Q))
// is 0, else -Q/2.  NARROW: q <= 31, so 32-bit words hold them.  A non-finite
// r gives NaN, as the fp64 form does.
template <bool NARROW>
__device__ inline double sym_digit(double r, int q) {
    const long long bits = __double_as_longlong(r);
    const int ex = (int)((bits >> 52) & 0x7ff);
    const long long m = (bits & 0xfffffffffffffll) | 0x10000000000000ll;   // |r| = m 2^-s
    const int s = 1075 - ex;
    // an integer: bits shifted out at the top are multiples of 2^64, above bit q
    unsigned long long u = s > 0 ? (unsigned long long)rne_shift(m, s)
                                 : (s > -64 ? (unsigned long long)m << -s : 0ull);
    u = bits < 0 ? 0ull - u : u;
    double d;
    if constexpr (NARROW) {
        const unsigned int w = (unsigned int)u << (31 - q);       // bits q .. 0 of u
        const int v = (int)(w << 1) >> (32 - q);
        d = double_of_bits(w == 0x40000000u ? -v : v);
    } else {
        const unsigned long long w = u << (63 - q);
        const long long v = (long long)(w << 1) >> (64 - q);
        d = double_of_bits(w == 0x4000000000000000ull ? -v : v);
    }
    return ex == 0x7ff ? __longlong_as_double(0x7ff8000000000000ll) : d;
}

// Asymmetric form: digit 0 = rint(x), then x <- Q (x - digit) for the next one.
// The remainder is kept as f 2^-s; x - rint(x) and the scaling by Q are exact
// in fp64 too, so both forms see the same x.
template <int N>
__device__ inline void asym_digits(double r, int q, double (&digit)[N]) {
    const long long bits = __double_as_longlong(r);
    const int ex = (int)((bits >> 52) & 0x7ff);
    long long f = (bits & 0xfffffffffffffll) | 0x10000000000000ll;
    f = bits < 0 ? -f : f;
    int s = 1075 - ex;
    const bool whole = s <= 0;              // an integer (or not finite): digit 0 is r itself
    if (ex == 0) f = 0;                     // zero or subnormal: every digit is zero
#pragma unroll
    for (int d = 0; d < N; ++d) {
        if (d == 0 && whole) {
            digit[0] = r;
            f = 0;
            s = 1;
        } else if (s > 0) {
            const long long v = rne_shift(f, s);
            digit[d] = double_of_bits(v);
            if (v) f -= v << s;             // v = 0 wherever s > 53
        } else {
            // at most Q/2 in magnitude
            digit[d] = double_of_bits(f << -s);
            f = 0;
            s = 1;
        }
        s -= q;
        if (f == 0) s = 1;
    }
    if (ex == 0x7ff) {
#pragma unroll
        for (int d = 1; d < N; ++d) digit[d] = __longlong_as_double(0x7ff8000000000000ll);
    }
}

}  // namespace tdg
