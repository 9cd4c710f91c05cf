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
//     largest are dropped, where an FP64 sum would round at 2^-53 of its partial sums. A block is one
//     sum's points along one grid line (grf_diffs.cuh), since across lines the magnitudes may differ by
//     more than that: what a derivative keeps depends on no point that it does not read;
//   * where the weights leave no room above G guard bits, sums are taken in halves, quarters and so on by constant
//     shifts of the terms, or the differences that are weighted are shifted right by what their own magnitude asks
//     for (fx_room): what that drops lies below 2^-53 of the largest term;
//   * the integer sums are independent of their order, so every caller gets the same bits;
//   * the sum times a positive constant (the grid-spacing factor, as a 64-bit mantissa) is rounded once to
//     double.
// Range: the caller bounds the block exponent (FxRange), so that no result leaves the normal doubles and no
// result has to be checked: blocks below the range count as their values' multiples of a tiny unit (2^-900
// and less at common spacings), blocks above it, with infinities and NaNs among them, take the FP64 sums.
// The functions compile for the host too, where tests compare them with exact arithmetic.
#pragma once

#include <cstring>

#include "grf_point.cuh"

namespace grf {

// A positive finite constant c = m 2^(e - 63), m with its top bit set.
struct FxScale {
    unsigned long long m;
    int e, zero;  // (no padding: descriptors that hold it are compared bytewise)
};

inline FxScale fx_scale_of(double c) {
    unsigned long long b;
    std::memcpy(&b, &c, sizeof b);
    FxScale s;
    s.e = (int)(b >> 52) - 1023;
    s.zero = 0;
    s.m = (b << 11) | 0x8000000000000000ull;
    return s;
}

// Block exponents whose results (sums of magnitude 2^0 .. 2^63 units, of 2^shift units where fx_room coarsens
// them, of 2^-25 units where fx_aligned refines them, times constants of exponents lo .. hi or 1) are normal
// doubles.
struct FxRange {
    int emin, emax;
};

inline FxRange fx_range(int lo, int hi, int shift = 0) {
    FxRange r;
    r.emin = 96 - (lo < 0 ? lo : 0);
    r.emax = 2046 - 13 - shift - (hi > 0 ? hi : 0);
    // no block qualifies: no exponent is left, or a constant is itself zero, subnormal or infinite (fx_scale_of holds
    // normal ones only)
    if (r.emin > r.emax || lo <= -1023 || hi >= 1024) r.emax = -1;
    return r;
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

// x in units of 2^(emax - 1075 - G), truncated towards zero, |result| < 2^(53 + G), for |x| of exponent at
// most emax; lim = fx_lim<G>(emax) is the exponent's word the shift is counted from.
template <int G>
GRF_HD int fx_lim(int emax) { return (int)((unsigned)(emax + 11 - G) << 20 | 0xfffffu); }

GRF_HD long long fx_int(double x, int lim) {
#ifdef __CUDA_ARCH__
    // 12 instructions: the shift count, the mantissa at the top of 64 bits, the shift (by 64 and more: to
    // zero), the sign
    const int hi = __double2hiint(x), lo = __double2loint(x);
    const unsigned s = (unsigned)(lim - (hi & 0x7fffffff)) >> 20;
    const unsigned uh = __funnelshift_l(lo, hi, 11) | 0x80000000u, ul = (unsigned)lo << 11;
    long long r;
    asm("{\n\t.reg .pred p;\n\t.reg .b64 u;\n\t"
        "mov.b64 u, {%2, %1};\n\tshr.u64 %0, u, %3;\n\tsetp.lt.s32 p, %4, 0;\n\t@p neg.s64 %0, %0;\n\t}"
        : "=&l"(r)
        : "r"(uh), "r"(ul), "r"(s), "r"(hi));
    return r;
#else
    const unsigned long long b = fx_bits(x);
    const unsigned s = (unsigned)(lim - ((int)(b >> 32) & 0x7fffffff)) >> 20;
    const unsigned long long u = (b << 11) | 0x8000000000000000ull;
    const long long r = s > 63 ? 0 : (long long)(u >> s);
    return (long long)b < 0 ? -r : r;
#endif
}

// |I| 2^z with the top bit set, and z (64 and 0 for I = 0).
GRF_HD unsigned long long fx_normal(long long I, int& z) {
#ifdef __CUDA_ARCH__
    unsigned long long u = (unsigned long long)I, r;
    asm("{\n\t.reg .pred p;\n\tsetp.lt.s64 p, %0, 0;\n\t@p neg.s64 %0, %0;\n\t}" : "+l"(u));
    z = __clzll((long long)u);
    asm("shl.b64 %0, %1, %2;" : "=l"(r) : "l"(u), "r"(z));
    return r;
#else
    const unsigned long long u = (unsigned long long)(I < 0 ? -I : I);
    z = u ? __builtin_clzll(u) : 64;
    return u ? u << z : 0;
#endif
}

// The top word of |x|, for x < 0 of |x| - 1: enough to bound |x|.
GRF_HD unsigned fx_top(long long x) {
    const int hi = (int)(x >> 32);
    return (unsigned)(hi ^ (hi >> 31));
}
GRF_HD int fx_clz32(unsigned x) {
#ifdef __CUDA_ARCH__
    return __clz((int)x);
#else
    return x ? __builtin_clz(x) : 32;
#endif
}
// The right shift (below 32) after which integers whose top words are OR-ed in `top` are below 2^bits.
GRF_HD int fx_room(unsigned top, int bits) { return fx_max(0, 64 - bits - fx_clz32(top)); }

// x >> s: for 0 <= s < 32, and for any s >= 0.
GRF_HD long long fx_sar(long long x, int s) {
#ifdef __CUDA_ARCH__
    const int hi = (int)(x >> 32);
    return ((long long)(hi >> s) << 32) | __funnelshift_r((unsigned)x, (unsigned)hi, (unsigned)s);
#else
    return x >> s;
#endif
}
GRF_HD long long fx_sar_any(long long x, int s) {
#ifdef __CUDA_ARCH__
    long long r;
    asm("shr.s64 %0, %1, %2;" : "=l"(r) : "l"(x), "r"(s));  // (clamped at 64)
    return r;
#else
    return x >> (s > 63 ? 63 : s);
#endif
}
// x in units of 2^e as an integer in units of 2^(E - left), e <= E, left <= 31: for n = left - (E - e), x << n or
// x >> -n.
GRF_HD long long fx_aligned(long long x, int n) {
#ifdef __CUDA_ARCH__
    const int l = fx_max(n, 0);
    const unsigned hi = __funnelshift_l((unsigned)x, (unsigned)((unsigned long long)x >> 32), (unsigned)l);
    x = (long long)(((unsigned long long)hi << 32) | ((unsigned)x << l));
    return fx_sar_any(x, fx_max(-n, 0));
#else
    return n >= 0 ? (long long)((unsigned long long)x << n) : fx_sar_any(x, -n);
#endif
}

// The double of mantissa p (64 bits, top bit set; rounded to nearest) and biased exponent E in the normal
// range, with the sign of I; 0 where z = 64.
GRF_HD double fx_pack(unsigned long long p, int E, int z, long long I) {
    const unsigned long long r = (p >> 11) + ((p >> 10) & 1ull);
    const unsigned eh = z == 64 ? 0u : (unsigned)(E - 1) << 20;
    const unsigned hi = (unsigned)(r >> 32) + eh;
    const unsigned sg = (unsigned)((unsigned long long)I >> 32) & 0x80000000u;
#ifdef __CUDA_ARCH__
    return __hiloint2double((int)(hi | sg), (int)(unsigned)r);
#else
    const unsigned long long b = ((unsigned long long)(hi | sg) << 32) | (unsigned)r;
    double x;
    std::memcpy(&x, &b, sizeof x);
    return x;
#endif
}

// I 2^(emax - 1075 - G), rounded to double.
template <int G>
GRF_HD double fx_value(long long I, int emax) {
    int z;
    const unsigned long long u = fx_normal(I, z);
    return fx_pack(u, emax - z + 11 - G, z, I);
}

// I 2^(emax - 1075 - G) times the constant c, rounded once to double.
template <int G>
GRF_HD double fx_value(long long I, int emax, const FxScale& c) {
    int z;
    const unsigned long long u = fx_normal(I, z);
#ifdef __CUDA_ARCH__
    unsigned long long p = __umul64hi(u, c.m);
#else
    unsigned long long p = (unsigned long long)(((unsigned __int128)u * c.m) >> 64);
#endif
    int E = emax + c.e - z + 12 - G;
    if (!(p >> 63)) {
        p += p;
        --E;
    }
    return fx_pack(p, E, z, I);
}

}  // namespace grf
