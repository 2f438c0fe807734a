// Device helpers of the fixed-point FP64 kernels: blocks in memory, the mixing
// tile, fifth-direction mixing and the epilogue's conversions (arithmetic in
// fixed.cuh, field layout in dwf_internal.h).
//
// A block field stores the field's 16-byte vectors with 64-bit integers in the
// place of the doubles, and one word of two exponents (fx_word) per (site, s),
// [site][Ls], behind it (FieldRef::fx).  Registers hold a block as 12 pairs in the
// order of the FP64 kernels (even pairs P_+, odd pairs P_-), so project() and
// reconstruct() of stencil.cuh apply to it once both halves have one exponent.
#pragma once

#include "fields.cuh"
#include "fixed.cuh"

namespace dwf {

template <> struct PairReal<longlong2> { typedef long long R; };
__device__ __forceinline__ longlong2 p_make(long long a, long long b) { return make_longlong2(a, b); }
__device__ __forceinline__ longlong2 p_splat(long long a) { return make_longlong2(a, a); }
__device__ __forceinline__ longlong2 p_fma(longlong2 a, longlong2 b, longlong2 c)
{
    return make_longlong2(a.x * b.x + c.x, a.y * b.y + c.y);
}
__device__ __forceinline__ longlong2 p_add(longlong2 a, longlong2 b) { return make_longlong2(a.x + b.x, a.y + b.y); }

namespace {

// ------------------------------------------------------------ blocks in memory
template <bool RO>
__device__ __forceinline__ void fx_ld(const FieldRef &f, size_t site, int s, int Ls, longlong2 *v)
{
    const longlong2 *p = reinterpret_cast<const longlong2 *>(f.v) + (site * 12) * Ls + s;
#pragma unroll
    for (int k = 0; k < 12; ++k) v[k] = RO ? __ldg(p + (size_t)k * Ls) : p[(size_t)k * Ls];
}
__device__ __forceinline__ void fx_st(const FieldRef &f, size_t site, int s, int Ls, const longlong2 *v, int e)
{
    longlong2 *p = reinterpret_cast<longlong2 *>(f.v) + (site * 12) * Ls + s;
#pragma unroll
    for (int k = 0; k < 12; ++k) p[(size_t)k * Ls] = v[k];
    f.fx[site * Ls + s] = e;
}

// the exponent (or mark) of the pairs of chirality CHI
template <int CHI>
__device__ __forceinline__ int fx_half_exponent(const double2 *v)
{
    uint32_t m = 0, low = 0;
#pragma unroll
    for (int k = CHI; k < 12; k += 2) {
        m = max(m, max((uint32_t)__double2hiint(v[k].x) & 0x7fffffffu, (uint32_t)__double2hiint(v[k].y) & 0x7fffffffu));
        low |= (uint32_t)__double2loint(v[k].x) | (uint32_t)__double2loint(v[k].y);
    }
    return fx_exponent(m, low);
}
// doubles -> integers of B bits below 2^e, e of each half (B = FX_BITS: of a field);
// a marked block keeps the doubles' bits.  Returns the exponents' word.
__device__ __forceinline__ int fx_pack(const double2 *v, int B, longlong2 *t)
{
    int ep = fx_half_exponent<0>(v), em = fx_half_exponent<1>(v);
    const bool raw = max(ep, em) == FX_RAW;
    if (B == FX_BITS) fx_near(ep, em);
#pragma unroll
    for (int k = 0; k < 12; ++k) {
        const int e = k & 1 ? em : ep;
        t[k] = raw ? make_longlong2(__double_as_longlong(v[k].x), __double_as_longlong(v[k].y))
                   : make_longlong2(fx_from_double(v[k].x, e, B), fx_from_double(v[k].y, e, B));
    }
    return raw ? FX_RAW_BLOCK : fx_word(ep, em);
}
// one value of a marked block, or of one whose exponent leaves FP64's normal range: out
// of line, as 24 inlined scalings would crowd the instruction cache
__device__ __noinline__ double fx_value_rare(long long r, int s, bool raw)
{
    return raw ? __longlong_as_double(r) : fx_to_double(r, s);
}
// v = r 2^(s0 or s1 by chirality), or the raw doubles
__device__ __forceinline__ void fx_to_doubles(const longlong2 *r, int s0, int s1, bool raw, double2 *v)
{
    if (!raw && fx_normal_shift(s0) && fx_normal_shift(s1)) {
#pragma unroll
        for (int k = 0; k < 12; ++k) {
            const int s = k & 1 ? s1 : s0;
            v[k] = make_double2(fx_to_double_normal(r[k].x, s), fx_to_double_normal(r[k].y, s));
        }
    } else {
#pragma unroll
        for (int k = 0; k < 12; ++k) {
            const int s = k & 1 ? s1 : s0;
            v[k] = make_double2(fx_value_rare(r[k].x, s, raw), fx_value_rare(r[k].y, s, raw));
        }
    }
}
// v[12] <- an FP64 or block field as doubles
template <bool RO>
__device__ __forceinline__ void fx_ld_double(const FieldRef &f, size_t site, int s, int Ls, double2 *v)
{
    if (f.fx) {
        longlong2 t[12];
        fx_ld<RO>(f, site, s, Ls, t);
        const int e = f.fx[site * Ls + s];
        fx_to_doubles(t, fx_half<0>(e) - FX_BITS, fx_half<1>(e) - FX_BITS, fx_is_raw(e), v);
    } else {
        ld_pairs<DWF_F64, RO>(f, site, s, Ls, v);
    }
}

// bits of the largest of the pairs of chirality CHI
template <int CHI>
__device__ __forceinline__ int fx_half_width(const longlong2 *v)
{
    uint32_t hi = 0, lo = 0;
#pragma unroll
    for (int k = CHI; k < 12; k += 2) {
        const longlong2 q = v[k];
        const int32_t hx = (int32_t)(q.x >> 32), hy = (int32_t)(q.y >> 32);
        hi |= (uint32_t)(hx ^ (hx >> 31)) | (uint32_t)(hy ^ (hy >> 31));
        lo |= (uint32_t)((int32_t)q.x ^ (hx >> 31)) | (uint32_t)((int32_t)q.y ^ (hy >> 31));
    }
    // a set of zeros and minus ones has no bits above the sign: one, so that fx_align shifts by at most 62
    const int w = hi ? 64 - __clz((int)hi) : 32 - __clz((int)lo);
    return w > 0 ? w : 1;
}
// all pairs of chirality CHI zero
template <int CHI>
__device__ __forceinline__ bool fx_half_zero(const longlong2 *v)
{
    unsigned long long any = 0;
#pragma unroll
    for (int k = CHI; k < 12; k += 2) any |= (unsigned long long)v[k].x | (unsigned long long)v[k].y;
    return any == 0;
}

// ------------------------------------------------------------------ the tile
// Tile rows of one (site, s): 12 vectors of 16 bytes, each two reals as limbs
// (low, high; radix 2^29), rows 13 vectors apart so that eight lanes' 16-byte
// accesses hit distinct banks; te[site row] the exponents' words.  A marked row
// holds raw doubles.
constexpr int FX_ROW = 13;
__host__ __device__ constexpr int fx_site_stride(int Ls) { return Ls * FX_ROW + 1; }

__device__ __forceinline__ void fx_put(int4 *row, const longlong2 *t, int e)
{
#pragma unroll
    for (int k = 0; k < 12; ++k) {
        int4 q;
        if (fx_is_raw(e)) {
            q = make_int4((int)t[k].x, (int)(t[k].x >> 32), (int)t[k].y, (int)(t[k].y >> 32));
        } else {
            fx_limbs29(t[k].x, q.x, q.y);
            fx_limbs29(t[k].y, q.z, q.w);
        }
        row[k] = q;
    }
}
__device__ __forceinline__ double fx_tile_double(int lo, int hi, int e, int chi, int B)
{
    return fx_is_raw(e) ? __hiloint2double(hi, lo)
                        : fx_to_double(((int64_t)hi << 29) + lo, (chi ? fx_half<1>(e) : fx_half<0>(e)) - B);
}

// A fifth-direction matrix: constants {mantissa low, high word, exponent, 0} of B
// bits, [chi][t][s], the same entries as doubles, and its kind.
struct FxMat {
    const int4 *c;
    const double *m;
    int band;   // 0 dense, 1 cyclic tridiagonal, 2 diagonal
};

// E[chi] of output s: the largest exponent of M_st x_t over the rows t; returns
// whether a row is marked.
__device__ __forceinline__ bool fx_mix_exponents(const FxMat &M, const int *te, int s, int Ls, int *E)
{
    const int n = M.band == 0 ? Ls : (M.band == 1 ? 3 : 1);
    int t = M.band == 1 ? (s ? s - 1 : Ls - 1) : s, mark = 0;
    const int4 *c = M.c + s;
    E[0] = E[1] = 2 * FX_ZERO;
#pragma unroll 4
    for (int i = 0; i < n; ++i) {
        const int e = te[t];
        mark = max(mark, e);
        E[0] = max(E[0], __ldg(&c[t * Ls].z) + fx_half<0>(e));
        E[1] = max(E[1], __ldg(&c[(Ls + t) * Ls].z) + fx_half<1>(e));
        t = t + 1 < Ls ? t + 1 : 0;
    }
    return fx_is_raw(mark);
}

// r[k] (pairs of chirality CHI only): (M tile)(s) = r 2^(E + 58 - 2 B).  Every product
// M_st x_t is taken against E by shifting the constant: a row of small half blocks
// keeps its bits where it meets the large ones of other rows.  Constants that vanish there are
// skipped, and those below 2^28 take one multiply-add instead of three: the
// inverse's entries fall off by a factor kappa per slice (0.023 for b 1.5, c 0.5).
// Lane s starts at row s, so that a warp meets constants of one size together.
template <int CHI>
__device__ __forceinline__ void fx_mix_chi(const FxMat &M, const int4 *tile, const int *te, int s, int Ls, int E,
                                           longlong2 *r)
{
    const int n = M.band == 0 ? Ls : (M.band == 1 ? 3 : 1);
    int t = M.band == 1 ? (s ? s - 1 : Ls - 1) : s;
    const int4 *c = M.c + CHI * Ls * Ls + s;
    const short *te2 = reinterpret_cast<const short *>(te) + CHI;   // one half of each word
    int64_t hh[12], x[12];
#pragma unroll
    for (int k = 0; k < 12; ++k) hh[k] = 0, x[k] = 1 << 28;   // the cross sums are rounded at 2^29
    int4 next = __ldg(&c[t * Ls]);   // the constant of one row ahead (K_a 492 -> 485 us, K_b 793 -> 778 at 16^3x32, Ls 16)
#pragma unroll 1
    for (int i = 0; i < n; ++i) {
        const int4 q = next;
        const int sh = E - (q.z + te2[2 * t]);
        const int4 *row = tile + t * FX_ROW + CHI;
        t = t + 1 < Ls ? t + 1 : 0;
        next = __ldg(&c[t * Ls]);
        if (sh >= 58) continue;
        const int64_t m = (((int64_t)q.y << 32) | (uint32_t)q.x) >> sh;
        if (sh >= 30) {   // the constant, below 2^28, is its low limb
#pragma unroll
            for (int k = 0; k < 6; ++k) {
                const int4 v = row[2 * k];
                x[2 * k] = fx_mad1(v.y, (int32_t)m, x[2 * k]);
                x[2 * k + 1] = fx_mad1(v.w, (int32_t)m, x[2 * k + 1]);
            }
            continue;
        }
        int32_t cl, ch;
        fx_limbs29(m, cl, ch);
#pragma unroll
        for (int k = 0; k < 6; ++k) {
            const int4 v = row[2 * k];
            fx_mad(v.x, v.y, cl, ch, hh[2 * k], x[2 * k]);
            fx_mad(v.z, v.w, cl, ch, hh[2 * k + 1], x[2 * k + 1]);
        }
    }
#pragma unroll
    for (int k = 0; k < 6; ++k)
        r[2 * k + CHI] = make_longlong2(hh[2 * k] + (x[2 * k] >> 29), hh[2 * k + 1] + (x[2 * k + 1] >> 29));
}

// the same product in FP64, for rows with non-finite entries: o = M tile
__device__ __noinline__ void fx_mix_raw(const FxMat &M, const int4 *tile, const int *te, int s, int Ls, int B, double2 *o)
{
    for (int k = 0; k < 12; ++k) o[k] = make_double2(0.0, 0.0);
    for (int t = 0; t < Ls; ++t) {
        const int dt = t - s < 0 ? t - s + Ls : t - s;
        if ((M.band == 1 && dt > 1 && dt < Ls - 1) || (M.band == 2 && dt != 0)) continue;
        for (int k = 0; k < 12; ++k) {
            const double m = M.m[(size_t)(k & 1) * Ls * Ls + (size_t)t * Ls + s];
            if (m == 0.0) continue;   // a row that the matrix does not couple
            const int4 q = tile[t * FX_ROW + k];
            o[k].x = fma(m, fx_tile_double(q.x, q.y, te[t], k & 1, B), o[k].x);
            o[k].y = fma(m, fx_tile_double(q.z, q.w, te[t], k & 1, B), o[k].y);
        }
    }
}

// A mixing's result: 12 pairs r of 2^(E[chi] + 58 - 2 B) or, where a row that enters
// holds non-finite values, the doubles' bits (raw).
struct FxSum {
    longlong2 r[12];
    int E[2];
    bool raw;
};
__device__ __forceinline__ void fx_mix(const FxMat &M, const int4 *tile, const int *te, int s, int Ls, int B, FxSum &S)
{
    S.raw = fx_mix_exponents(M, te, s, Ls, S.E);
    if (S.raw) {
        double2 o[12];
        fx_mix_raw(M, tile, te, s, Ls, B, o);
#pragma unroll
        for (int k = 0; k < 12; ++k) S.r[k] = make_longlong2(__double_as_longlong(o[k].x), __double_as_longlong(o[k].y));
        return;
    }
    fx_mix_chi<0>(M, tile, te, s, Ls, S.E[0], S.r);
    fx_mix_chi<1>(M, tile, te, s, Ls, S.E[1], S.r);
}
__device__ __forceinline__ void fx_sum_doubles(const FxSum &S, int B, double2 *o)
{
    fx_to_doubles(S.r, S.E[0] + 58 - 2 * B, S.E[1] + 58 - 2 * B, S.raw, o);
}
// S += T; both below 2^62 in magnitude, and so is the sum
__device__ __forceinline__ void fx_sum_add(FxSum &S, const FxSum &T, int B)
{
    if (S.raw || T.raw) {
#pragma unroll
        for (int k = 0; k < 12; ++k) {
            const int a = S.E[k & 1] + 58 - 2 * B, b = T.E[k & 1] + 58 - 2 * B;
            const double2 q = make_double2(fx_value_rare(S.r[k].x, a, S.raw) + fx_value_rare(T.r[k].x, b, T.raw),
                                           fx_value_rare(S.r[k].y, a, S.raw) + fx_value_rare(T.r[k].y, b, T.raw));
            S.r[k] = make_longlong2(__double_as_longlong(q.x), __double_as_longlong(q.y));
        }
        S.raw = true;
        return;
    }
#pragma unroll
    for (int c = 0; c < 2; ++c) {
        const int E = max(S.E[c], T.E[c]) + 1, a = min(E - S.E[c], 63), b = min(E - T.E[c], 63);
        S.E[c] = E;
#pragma unroll
        for (int k = c; k < 12; k += 2)
            S.r[k] = make_longlong2((S.r[k].x >> a) + (T.r[k].x >> b), (S.r[k].y >> a) + (T.r[k].y >> b));
    }
}

// out(site, s) <- the doubles o, as an FP64 or a block field
__device__ __forceinline__ void fx_store_double(const FieldRef &out, size_t site, int s, int Ls, const double2 *o)
{
    if (out.fx) {
        longlong2 t[12];
        const int e = fx_pack(o, FX_BITS, t);
        fx_st(out, site, s, Ls, t, e);
    } else {
        st_pairs<DWF_F64>(out, site, s, Ls, o);
    }
}
// out(site, s) <- S
__device__ __forceinline__ void fx_store_sum(const FieldRef &out, size_t site, int s, int Ls, FxSum &S, int B)
{
    if (!out.fx || S.raw) {
        double2 o[12];
        fx_sum_doubles(S, B, o);
        fx_store_double(out, site, s, Ls, o);
        return;
    }
    const int wp = fx_half_width<0>(S.r), wm = fx_half_width<1>(S.r);
    // |value| < 2^top
    const int tp = fx_half_zero<0>(S.r) ? FX_ZERO : wp + S.E[0] + 58 - 2 * B;
    const int tm = fx_half_zero<1>(S.r) ? FX_ZERO : wm + S.E[1] + 58 - 2 * B;
    int ep = tp, em = tm;
    fx_near(ep, em);
#pragma unroll
    for (int k = 0; k < 12; ++k) {
        const int w = k & 1 ? wm : wp, down = 63 - FX_BITS + (k & 1 ? em - tm : ep - tp);
        S.r[k] = make_longlong2(fx_align(S.r[k].x, w, down), fx_align(S.r[k].y, w, down));
    }
    fx_st(out, site, s, Ls, S.r, fx_word(ep, em));
}

}  // namespace
}  // namespace dwf
