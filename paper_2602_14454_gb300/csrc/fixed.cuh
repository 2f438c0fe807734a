// Block fixed-point arithmetic for the FP64 operator.
//
// GB300 issues two FP64 operations per clock and SM (measured: 1.98 DFMA lanes) but
// about 32 integer multiply-adds 32 x 32 + 64 -> 64 (the counters show four cycles
// of the multiply pipe per warp), so the products of the FP64 hop and of its
// fifth-direction mixing run on the integer pipe.  A block is the 24 reals x_k of one (site, s):
//     x_k = F_k 2^(e - 59),  F_k integers below 2^59 in magnitude,
// e the block's exponent (every |x_k| < 2^e, the largest at least 2^(e - 1)).
// A product takes two limbs per factor and three multiply-adds (hi hi and the two
// cross products; lo lo lies below the kept bits), sums are exact integer
// additions, and one rounding to FP64 follows at the end.  Where FP64 keeps 53
// bits of every number, a block keeps 59 bits relative to its largest: its
// rounding errors are the smaller ones in the norm of every (site, s).
//
// A block with an infinite or NaN entry is marked by e = FX_RAW and holds the
// doubles' own bits; a kernel that reads a marked block computes the sites it
// reaches in FP64, so non-finite values spread as FP64 arithmetic spreads them.
//
// Everything here is 64-bit integer C++ that also runs on the host.
#pragma once

#include <cmath>
#include <cstdint>
#include <cstring>

#if defined(__CUDACC__)
#define FX_HD __host__ __device__ __forceinline__
#else
#define FX_HD inline
#endif

namespace dwf {

constexpr int FX_BITS = 59;
constexpr int FX_RAW = 0x4000;     // the block holds raw doubles
constexpr int FX_ZERO = -0x4000;   // every entry is zero

// Bits of a mixing tile's entries and of the mixing constants: the sums over Ls
// slices of hi hi and of the cross products (radix 2^29) stay below 2^63.
FX_HD constexpr int fx_mix_bits(int Ls) { return Ls <= 16 ? 58 : 57; }

FX_HD int64_t fx_bits_of(double x)
{
#if defined(__CUDA_ARCH__)
    return __double_as_longlong(x);
#else
    int64_t b;
    std::memcpy(&b, &x, 8);
    return b;
#endif
}
FX_HD double fx_of_bits(int64_t b)
{
#if defined(__CUDA_ARCH__)
    return __longlong_as_double(b);
#else
    double x;
    std::memcpy(&x, &b, 8);
    return x;
#endif
}
// number of leading zeros; 64 for 0
FX_HD int fx_clz(uint64_t x)
{
#if defined(__CUDA_ARCH__)
    return __clzll((long long)x);
#else
    return x ? __builtin_clzll(x) : 64;
#endif
}

// R 2^s as a double for -1000 < s < 950, where it is normal, rounded once to nearest
// even.  In integers: the conversion instruction runs on the FP64 pipe.
FX_HD constexpr bool fx_normal_shift(int s) { return s > -1000 && s < 950; }
FX_HD double fx_to_double_normal(int64_t R, int s)
{
    const uint64_t sg = (uint64_t)(R >> 63), a = ((uint64_t)R ^ sg) - sg;
    const int z = fx_clz(a);
    const uint64_t v = a << ((z - 1) & 63);   // leading bit at 62
    const uint64_t r = (v + 0x1ff + ((v >> 10) & 1)) >> 10;
    const uint64_t e = (uint64_t)(uint32_t)(1085 + s - z) << 52;   // r's bit 52 adds the last one
    return fx_of_bits(a ? (int64_t)((e + r) | (sg << 63)) : 0);
}
// any s (rounded twice below FP64's normal range)
FX_HD double fx_to_double(int64_t R, int s)
{
    return fx_normal_shift(s) ? fx_to_double_normal(R, s) : scalbn((double)R, s);
}

// The exponent field of the largest of the doubles whose high words' magnitudes
// have the maximum m; `low`: the bitwise or of all their low words.
// FX_RAW / FX_ZERO, or e with |x| < 2^e.
FX_HD int fx_exponent(uint32_t m, uint32_t low)
{
    const int eb = (int)(m >> 20);
    if (eb == 0x7ff) return FX_RAW;
    if (m == 0 && low == 0) return FX_ZERO;
    return (eb > 1 ? eb : 1) - 1022;
}

// x 2^(B - e) truncated to an integer, |x| < 2^e, B >= 53
FX_HD int64_t fx_from_double(double x, int e, int B)
{
    const int64_t b = fx_bits_of(x);
    const int32_t hi = (int32_t)(b >> 32);
    const int ex = (int)(((uint32_t)hi >> 20) & 0x7ffu);
    const uint32_t mh = ((uint32_t)hi & 0xfffffu) | (ex ? 0x100000u : 0u);
    int d = e + 1022 - (ex ? ex : 1);
    d = d > 63 ? 63 : d < 0 ? 0 : d;   // d < 0 only where e is a mark
    const uint64_t M = (((uint64_t)mh << 32 | (uint32_t)b) << (B - 53)) >> d;
    const int64_t sg = (int64_t)(hi >> 31);
    return ((int64_t)M ^ sg) - sg;
}

// Limbs in radix 2^31, x = h 2^31 + l: with the low one in [0, 2^31) (two
// instructions) ...
FX_HD void fx_limbs31(int64_t x, int32_t &l, int32_t &h)
{
    l = (int32_t)((uint32_t)x & 0x7fffffffu);
    h = (int32_t)(x >> 31);
}
// ... or in [-2^30, 2^30), so that either limb can be negated and the dropped
// products lo lo with the first kind average to zero
FX_HD void fx_limbs31s(int64_t x, int32_t &l, int32_t &h)
{
    l = (int32_t)((uint32_t)x << 1) >> 1;
    h = (int32_t)((x + (1 << 30)) >> 31);
}
// Limbs in radix 2^29, the low one signed
FX_HD void fx_limbs29(int64_t x, int32_t &l, int32_t &h)
{
    l = (int32_t)((uint32_t)x << 3) >> 3;
    h = (int32_t)((x + (1 << 28)) >> 29);
}

// c + a b, one multiply-add.  In PTX: from C++ the compiler forms 64-bit products of
// the sign-extended limbs, several instructions each.
FX_HD int64_t fx_mad1(int32_t a, int32_t b, int64_t c)
{
#if defined(__CUDA_ARCH__)
    int64_t r;
    asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(r) : "r"(a), "r"(b), "l"(c));
    return r;
#else
    return c + (int64_t)a * b;
#endif
}
// one product's three multiply-adds
FX_HD void fx_mad(int32_t al, int32_t ah, int32_t bl, int32_t bh, int64_t &hh, int64_t &x)
{
    hh = fx_mad1(ah, bh, hh);
    x = fx_mad1(ah, bl, x);
    x = fx_mad1(al, bh, x);
}

// the leading position of a set of integers from the or of their (v ^ (v >> 63)): |v| < 2^bits
FX_HD int fx_width(uint64_t any) { return 64 - fx_clz(any); }
// v 2^(63 - bits) 2^-(down): v's leading bit moved to bit 62, then shifted down
FX_HD int64_t fx_align(int64_t v, int bits, int down)
{
    return (int64_t)((uint64_t)v << (63 - bits)) >> (down > 63 ? 63 : down);
}

}  // namespace dwf
