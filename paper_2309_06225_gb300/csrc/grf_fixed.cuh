// Stencil sums in block fixed point: integer arithmetic in place of FP64 for sums of grid values with
// small integer weights.
//
// GB300 executes 2 FP64 lanes per SM and clock against 64 integer lanes: one FP64 add occupies its pipe
// for 16-20 clocks a warp, a 64-bit integer add for about one, and the two run side by side. A
// finite-difference or dissipation sum over the points of one field is therefore taken in 64-bit
// integers, in units set by the largest magnitude among its own points, and rounded once:
//   * every value x of the block becomes the two's complement integer x / 2^(emax - 1075 - G), emax the
//     largest biased exponent of the block and G guard bits below the largest value's last bit. Values
//     down to 2^-G of the largest keep all their bits; of smaller ones the bits below 2^-(52 + G) of the
//     largest are dropped, where an FP64 sum would round at 2^-53 of its partial sums;
//   * sums with weights of total magnitude below 2^(10 - G) cannot overflow, and are exact and
//     independent of their order, so every caller gets the same bits;
//   * the sum times a positive constant (the grid-spacing factor, as a 64-bit mantissa) is rounded once to
//     double.
// A block whose values are all below 2^-959 counts as zeros below 2^-1013. An infinity or NaN among the
// block's values gives a NaN.
// The functions compile for the host too, where tests compare them with exact arithmetic.
#pragma once

#include <cstring>

#include "grf_point.cuh"

namespace grf {

// A positive finite constant c = m 2^(e - 63), m with its top bit set.
struct FxScale {
    unsigned long long m;
    int e;
};

inline FxScale fx_scale_of(double c) {
    unsigned long long b;
    std::memcpy(&b, &c, sizeof b);
    FxScale s;
    s.e = (int)(b >> 52) - 1023;
    s.m = (b << 11) | 0x8000000000000000ull;
    return s;
}

GRF_HD unsigned long long fx_bits(double x) {
#ifdef __CUDA_ARCH__
    return (unsigned long long)__double_as_longlong(x);
#else
    unsigned long long b;
    std::memcpy(&b, &x, sizeof b);
    return b;
#endif
}

// The top word of |x|; the largest one of a block gives its exponent.
GRF_HD int fx_mag(double x) { return (int)(fx_bits(x) >> 32) & 0x7fffffff; }
GRF_HD int fx_max(int a, int b) { return a > b ? a : b; }

constexpr int kFxNan = 1 << 20;  // "exponent" of a block that holds an infinity or a NaN

GRF_HD int fx_exponent(int mag) {
    const int e = mag >> 20;
    return e >= 2047 ? kFxNan : fx_max(e, 64);
}

// x in units of 2^(emax - 1075 - G), truncated towards zero; |result| < 2^(53 + G).
template <int G>
GRF_HD long long fx_int(double x, int emax) {
    const unsigned long long b = fx_bits(x);
    const int hi = (int)(b >> 32);
    int s = emax - ((hi & 0x7fffffff) >> 20);
    s = s < 63 ? s : 63;
    const unsigned long long m = (((b & 0x000fffffffffffffull) | 0x0010000000000000ull) << G) >> s;
    return hi < 0 ? -(long long)m : (long long)m;
}

// 2^E (1.f) with 64-bit mantissa p (top bit set) and biased exponent E, rounded to nearest; the sign of I.
GRF_HD double fx_pack(unsigned long long p, int E, long long I) {
    unsigned long long b = (p >> 11) + ((p >> 10) & 1ull) + ((unsigned long long)(unsigned)(E - 1) << 52);
    if (!((unsigned)(E - 1) < 2046u && I != 0)) {
        if (E > (kFxNan >> 1)) b = 0x7ff8000000000000ull;
        else b = (E > 0 && I != 0) ? 0x7ff0000000000000ull : 0ull;
    }
    b |= (unsigned long long)I & 0x8000000000000000ull;
#ifdef __CUDA_ARCH__
    return __longlong_as_double((long long)b);
#else
    double x;
    std::memcpy(&x, &b, sizeof x);
    return x;
#endif
}

GRF_HD int fx_clz(unsigned long long u) {
#ifdef __CUDA_ARCH__
    return __clzll((long long)u) & 63;
#else
    return u ? __builtin_clzll(u) : 0;
#endif
}

// I 2^(emax - 1075 - G), rounded to double.
template <int G>
GRF_HD double fx_value(long long I, int emax) {
    unsigned long long u = (unsigned long long)(I < 0 ? -I : I);
    const int z = fx_clz(u);
    u <<= z;
    return fx_pack(u, emax - z + 11 - G, I);
}

// I 2^(emax - 1075 - G) times the constant c, rounded once to double.
template <int G>
GRF_HD double fx_value(long long I, int emax, const FxScale& c) {
    unsigned long long u = (unsigned long long)(I < 0 ? -I : I);
    const int z = fx_clz(u);
    u <<= z;
#ifdef __CUDA_ARCH__
    unsigned long long p = __umul64hi(u, c.m);
#else
    unsigned long long p = (unsigned long long)(((unsigned __int128)u * c.m) >> 64);
#endif
    const int q = 1 - (int)(p >> 63);
    p <<= q;
    return fx_pack(p, emax + c.e - z - q + 12 - G, I);
}

}  // namespace grf
