// Block fixed-point arithmetic for the FP64 operator.
//
// GB300 issues two FP64 operations per clock and SM (measured: 1.98 DFMA lanes) but
// about 32 integer multiply-adds 32 x 32 + 64 -> 64 (the counters show four cycles
// of the multiply pipe per warp), so the products of the FP64 hop and of its
// fifth-direction mixing run on the integer pipe.  A block is the 24 reals of one
// (site, s), in two halves by chirality, P_+ and P_- (12 reals each: the fifth
// direction's matrices mix slices of one chirality and never the two):
//     x_k = F_k 2^(e - 59),  F_k integers below 2^59 in magnitude,
// e the half's exponent (every |x_k| < 2^e, the largest at least 2^(e - 1); in fields
// at least 2^(e - 5), see fx_near).
// A product takes two limbs per factor and three multiply-adds (hi hi and the two
// cross products; lo lo lies below the kept bits), sums are exact integer
// additions, and one rounding to FP64 follows at the end.
//
// Accuracy: FP64 keeps 53 bits of every number, a half block 55 to 59 bits relative to
// its largest.  Its errors are the smaller ones wherever the terms of an output are of
// the half blocks' size, so in the norm of every half block for links that mix
// colours; an entry 2^-k below the largest of its own half block keeps k bits less.
// Products that must keep entries of one half block apart by more than that (unit
// links, colours of very different size) take the FP64 kernels (hop variant 0).
//
// A block with an infinite or NaN entry is marked by e = FX_RAW in both halves and
// holds the doubles' own bits; a kernel that reads a marked block computes the sites it
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

// The exponents of a block's halves in one word, P_+ in the low 16 bits.  Doubles,
// links and constants have exponents within 1100; two hops with their mixings (no
// field is held in blocks for longer) stay within 6000, so no exponent comes near the
// marks, and marked words compare above all others.
FX_HD constexpr int fx_word(int ep, int em) { return (int)((uint32_t)em << 16 | ((uint32_t)ep & 0xffffu)); }
template <int CHI>
FX_HD constexpr int fx_half(int word) { return CHI ? word >> 16 : (int)(int16_t)(uint16_t)(uint32_t)word; }
constexpr int FX_RAW_BLOCK = fx_word(FX_RAW, FX_RAW);
FX_HD constexpr bool fx_is_raw(int word) { return word >= FX_RAW_BLOCK - FX_RAW; }

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
// Halves of a field whose exponents differ by at most 4 take the larger one: the other
// half keeps 55 bits or more, and a hop, which adds the two halves, need not shift them
// against one another (even-odd application at 16^3x32, Ls 16: 1229 us, and 1275 us
// where every block's halves lie 20 bits apart).
constexpr int FX_NEAR = 4;
FX_HD void fx_near(int &ep, int &em)
{
    const int top = ep > em ? ep : em;
    if (top - ep <= FX_NEAR && top - em <= FX_NEAR) ep = em = top;
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
