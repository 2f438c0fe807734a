// Canonical complex-double fields <-> internal halves, the links' copies and the
// 5D source of a 4D source.  All of it is bound by memory: every kernel here moves
// its canonical side in whole runs of sites and transposes through shared memory,
// where a thread per (site, s) on the canonical side would touch 192 bytes of its
// own per lane.  Even-odd FP32 at 32^3x64, Ls 16: pack with the first mixing 1214 us
// for 6.4 GB (1830 + 607 us as two strided kernels), unpack 800 us for 4.8 GB (1830);
// the links at 24^3x48 570 us for 2.1 GB (1647).
#include "fx_fields.cuh"

namespace dwf {
namespace {

// ------------------------------------------------------------------ packing
constexpr int kPackThreads = 128;
constexpr int kRow = 25;   // doubles per (site, s) in shared memory: odd, so 16 lanes along s hit distinct banks

// Canonical side of a CTA's tile: sites c0 .. c0 + nc - 1 of n, all slices, as
// 16-byte vectors; at most 12 per thread, all in flight at once.
template <bool STORE>
__device__ __forceinline__ void move_canonical(double *canon, double *buf, int n, int c0, int nc, int Ls, int tid)
{
    const int run = nc * 12, total = run * Ls;
    const float inv = 1.f / (float)run;
    double2 q[12];
#pragma unroll
    for (int j = 0; j < 12; ++j) {
        const int f = tid + j * kPackThreads;
        if (f >= total) break;
        const int s = (int)(((float)f + 0.5f) * inv), r = f - s * run, site = r / 12, k = r - site * 12;
        double2 *c = reinterpret_cast<double2 *>(canon) + ((size_t)s * n + c0) * 12 + r;
        const double *b = buf + (site * Ls + s) * kRow + 2 * k;
        if (STORE) __stcs(c, make_double2(b[0], b[1]));
        else q[j] = __ldcs(c);
    }
    if (STORE) return;
#pragma unroll
    for (int j = 0; j < 12; ++j) {
        const int f = tid + j * kPackThreads;
        if (f >= total) break;
        const int s = (int)(((float)f + 0.5f) * inv), r = f - s * run, site = r / 12, k = r - site * 12;
        double *b = buf + (site * Ls + s) * kRow + 2 * k;
        b[0] = q[j].x;
        b[1] = q[j].y;
    }
}

// the pairs of one (site, s) from a row of the buffer
template <typename T2>
__device__ __forceinline__ void row_pairs(const double *b, T2 *v)
{
    typedef typename PairReal<T2>::R R;
#pragma unroll
    for (int p = 0; p < 12; ++p) v[p] = p_make((R)b[canon_of_internal(2 * p)], (R)b[canon_of_internal(2 * p + 1)]);
}

// A CTA holds nc consecutive canonical sites x Ls slices.  FULL: sites of both
// parities (the sites 2 i and 2 i + 1 have index i in their halves), else the sites
// of one half, `even`.  On the internal side one thread takes a (site, s).
template <int P, bool FULL, bool UNPACK>
__global__ void __launch_bounds__(kPackThreads) pack_kernel(double *canon, FieldRef even, FieldRef odd,
                                                             const int *eo2lex, int n, int Ls, int NC)
{
    extern __shared__ __align__(16) double buf[];
    const int c0 = blockIdx.x * NC, nc = min(NC, n - c0), tid = threadIdx.x;
    if (!UNPACK) {
        move_canonical<false>(canon, buf, n, c0, nc, Ls, tid);
        __syncthreads();
    }
    if (tid < nc * Ls) {
        const int site = tid / Ls, s = tid - site * Ls, lex = c0 + site;
        const size_t i = FULL ? lex >> 1 : lex;
        const FieldRef &f = FULL && lex != __ldg(eo2lex + i) ? odd : even;
        double *b = buf + tid * kRow;
        double2 v[12];
        if (UNPACK) {
            ld_pairs_cs<P>(f, i, s, Ls, v);
#pragma unroll
            for (int p = 0; p < 12; ++p) {
                b[canon_of_internal(2 * p)] = v[p].x;
                b[canon_of_internal(2 * p + 1)] = v[p].y;
            }
        } else {
            row_pairs(b, v);
            bool done = false;
            if constexpr (P == DWF_F64) {
                if (f.fx) {   // as blocks
                    longlong2 t[12];
                    const int e = fx_pack(v, FX_BITS, t);
                    fx_st(f, i, s, Ls, t, e);
                    done = true;
                }
            }
            if (!done) st_pairs<P>(f, i, s, Ls, v);
        }
    }
    if (UNPACK) {
        __syncthreads();
        move_canonical<true>(canon, buf, n, c0, nc, Ls, tid);
    }
}

// Pack of an even-odd field with the first mixing of its application: x = canonical,
// xh = M x (a block field for FP64, dense or banded in FP32 for the others), which
// saves reading x again.
template <int P>
__global__ void __launch_bounds__(kPackThreads) pack_mix_kernel(const double *canon, FieldRef x, const MixArgs a, int NC)
{
    extern __shared__ __align__(16) double buf[];
    const int Ls = a.Ls, c0 = blockIdx.x * NC, nc = min(NC, a.Vh - c0), tid = threadIdx.x;
    const int site = tid / Ls, s = tid - site * Ls;
    const bool active = tid < nc * Ls;
    const size_t i = (size_t)c0 + site;
    move_canonical<false>(const_cast<double *>(canon), buf, a.Vh, c0, nc, Ls, tid);
    if constexpr (P == DWF_F64) {
        const int B = fx_mix_bits(Ls);
        int4 *tiles = reinterpret_cast<int4 *>(buf);   // over the buffer, whose rows are in registers by then
        int *te = reinterpret_cast<int *>(buf + (size_t)NC * max(Ls * kRow, fx_site_stride(Ls) * 2)) + site * Ls;
        int4 *tile = tiles + site * fx_site_stride(Ls);
        __syncthreads();
        longlong2 t[12];
        int e = 0;
        if (active) {
            double2 v[12];
            row_pairs(buf + tid * kRow, v);
            st_pairs<P>(x, i, s, Ls, v);
            e = fx_pack(v, B, t);
        }
        __syncthreads();
        if (active) {
            fx_put(tile + s * FX_ROW, t, e);
            te[s] = e;
        }
        __syncthreads();
        if (active) {
            FxSum S;
            fx_mix(FxMat{a.mat_fx, reinterpret_cast<const double *>(a.mat), a.band}, tile, te, s, Ls, B, S);
            fx_store_sum(a.out, i, s, Ls, S, B);
        }
    } else {
        const int tstride = Ls * 12 + 2;
        float2 *tiles = reinterpret_cast<float2 *>(buf);   // over the buffer as well
        float *mtx = reinterpret_cast<float *>(buf + (size_t)NC * Ls * kRow);
        for (int k = tid; k < 2 * Ls * Ls; k += kPackThreads) mtx[k] = reinterpret_cast<const float *>(a.mat)[k];
        __syncthreads();
        float2 v[12];
        if (active) {
            row_pairs(buf + tid * kRow, v);
            st_pairs<P>(x, i, s, Ls, v);
            if constexpr (P == DWF_F16) ld_pairs<P, false>(x, i, s, Ls, v);   // what the stored field holds
        }
        __syncthreads();
        float2 *tile = tiles + site * tstride;
        if (active) {
#pragma unroll
            for (int k = 0; k < 12; ++k) tile[s * 12 + k] = v[k];
        }
        __syncthreads();
        if (active) {
            float2 o[1][12];
#pragma unroll
            for (int k = 0; k < 12; ++k) o[0][k] = make_float2(0.f, 0.f);
            if (a.band) mix_pairs_band<1>(mtx, tile, s, Ls, o);
            else mix_pairs<1>(mtx, tile, s, Ls, o);
            st_pairs<P>(a.out, i, s, Ls, o[0]);
        }
    }
}

template <int P>
cudaError_t launch_pack_mix_p(const double *canon, FieldRef x, const MixArgs &a, cudaStream_t st)
{
    const int NC = kPackThreads / a.Ls;
    const size_t row = (size_t)a.Ls * kRow * sizeof(double), tile = (size_t)fx_site_stride(a.Ls) * sizeof(int4);
    const size_t smem = P == DWF_F64 ? NC * ((row > tile ? row : tile) + a.Ls * sizeof(int))
                                     : NC * row + (size_t)2 * a.Ls * a.Ls * sizeof(float);
    pack_mix_kernel<P><<<(a.Vh + NC - 1) / NC, kPackThreads, smem, st>>>(canon, x, a, NC);
    return cudaGetLastError();
}

template <bool FULL, bool UNPACK>
cudaError_t launch_pack(int prec, const double *canon, FieldRef even, FieldRef odd, const int *eo2lex, int n, int Ls,
                        cudaStream_t st)
{
    const int NC = FULL ? (kPackThreads / Ls) & ~1 : kPackThreads / Ls;   // at least 4 (Ls <= 32)
    const size_t smem = (size_t)NC * Ls * kRow * sizeof(double);
    const int g = (n + NC - 1) / NC;
    double *c = const_cast<double *>(canon);
    switch (prec) {
    case DWF_F64: pack_kernel<DWF_F64, FULL, UNPACK><<<g, kPackThreads, smem, st>>>(c, even, odd, eo2lex, n, Ls, NC); break;
    case DWF_F32: pack_kernel<DWF_F32, FULL, UNPACK><<<g, kPackThreads, smem, st>>>(c, even, odd, eo2lex, n, Ls, NC); break;
    case DWF_F16: pack_kernel<DWF_F16, FULL, UNPACK><<<g, kPackThreads, smem, st>>>(c, even, odd, eo2lex, n, Ls, NC); break;
    default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

// -------------------------------------------------------------------- links
struct Dims {
    int d[4];
    int bc[4];
};
constexpr int kLinks = 128;   // links per CTA: 16 sites of one parity, 8 directions

// A link for the fixed-point hop: entries U 2^(e - 59) as limbs {re low, re high, im
// low, im high} (fx_limbs31s), nine per link, and its exponent or mark.
__device__ __forceinline__ int link_exponent(const double2 *u)
{
    uint32_t m = 0, low = 0;
#pragma unroll
    for (int k = 0; k < 9; ++k) {
        m = max(m, max((uint32_t)__double2hiint(u[k].x) & 0x7fffffffu, (uint32_t)__double2hiint(u[k].y) & 0x7fffffffu));
        low |= (uint32_t)__double2loint(u[k].x) | (uint32_t)__double2loint(u[k].y);
    }
    return fx_exponent(m, low);
}
__device__ __forceinline__ int4 link_limbs(double2 q, int e)
{
    int4 w;
    fx_limbs31s(fx_from_double(q.x, e, FX_BITS), w.x, w.y);
    fx_limbs31s(fx_from_double(q.y, e, FX_BITS), w.z, w.w);
    return w;
}
// the same from an FP64 copy (a slab's)
__global__ void __launch_bounds__(128) links_to_limbs_kernel(const double2 *g64, int4 *gfx, int *ge, size_t n)
{
    for (size_t l = blockIdx.x * (size_t)blockDim.x + threadIdx.x; l < n; l += (size_t)gridDim.x * blockDim.x) {
        double2 u[9];
#pragma unroll
        for (int k = 0; k < 9; ++k) u[k] = g64[l * 9 + k];
        const int e = link_exponent(u);
        ge[l] = e;
#pragma unroll
        for (int k = 0; k < 9; ++k) gfx[l * 9 + k] = link_limbs(u[k], e);
    }
}

// Neighbouring CTAs take the two parities of the same sites, so that most of a
// link's second read (it belongs to both of its ends) comes from L2.
__global__ void __launch_bounds__(kLinks) pack_gauge_kernel(const double *U, Dims D, int Vh, double2 *g64, float4 *g32,
                                                            uint4 *g16, int4 *gfx, int *ge)
{
    __shared__ __align__(16) double2 u[kLinks * 9];
    __shared__ const double2 *from[kLinks];
    __shared__ bool minus[kLinks];   // the boundary phase is -1
    __shared__ bool dagger[kLinks];
    __shared__ int eu[kLinks];
    const int par = blockIdx.x & 1, tid = threadIdx.x;
    const long long first = (long long)(blockIdx.x >> 1) * kLinks, total = (long long)Vh * 8;
    const int n = (int)min((long long)kLinks, total - first);
    if (tid < n) {
        const int dir = (int)((first + tid) & 7), i = (int)((first + tid) >> 3), mu = dir & 3;
        const int hx = D.d[0] / 2;
        int c[4], r = i / hx;
        c[1] = r % D.d[1];
        r /= D.d[1];
        c[2] = r % D.d[2];
        c[3] = r / D.d[2];
        c[0] = 2 * (i - (i / hx) * hx) + ((c[1] + c[2] + c[3] + par) & 1);
        const bool fwd = dir < 4;
        const bool crosses = c[mu] == (fwd ? D.d[mu] - 1 : 0);
        if (!fwd) c[mu] = c[mu] ? c[mu] - 1 : D.d[mu] - 1;
        const size_t lex = c[0] + (size_t)D.d[0] * (c[1] + (size_t)D.d[1] * (c[2] + (size_t)D.d[2] * c[3]));
        from[tid] = reinterpret_cast<const double2 *>(U) + ((size_t)mu * 2 * Vh + lex) * 9;
        minus[tid] = crosses && D.bc[mu] < 0;
        dagger[tid] = !fwd;
    }
    __syncthreads();
    double2 in[9];   // all of a thread's loads in flight at once
#pragma unroll
    for (int j = 0; j < 9; ++j) {
        const int f = tid + j * kLinks, l = f / 9;
        if (f < n * 9) in[j] = __ldg(from[l] + (f - l * 9));
    }
#pragma unroll
    for (int j = 0; j < 9; ++j) {
        const int f = tid + j * kLinks, l = f / 9, k = f - l * 9, a = k / 3, b = k - a * 3;
        if (f >= n * 9) break;
        const bool m = minus[l];
        const double2 q = make_double2(m ? -in[j].x : in[j].x, m ? -in[j].y : in[j].y);
        if (dagger[l]) u[l * 9 + b * 3 + a] = make_double2(q.x, -q.y);
        else u[f] = q;
    }
    __syncthreads();
    const size_t out = (size_t)par * total + first;   // this CTA's first link
    if (tid < n) {
        eu[tid] = link_exponent(u + tid * 9);
        ge[out + tid] = eu[tid];
    }
    __syncthreads();
#pragma unroll
    for (int j = 0; j < 9; ++j) {
        const int f = tid + j * kLinks;
        if (f < n * 9) gfx[out * 9 + f] = link_limbs(u[f], eu[f / 9]);
    }
#pragma unroll
    for (int j = 0; j < 9; ++j) {
        const int f = tid + j * kLinks;
        if (f < n * 9) g64[out * 9 + f] = u[f];
    }
    for (int f = tid; f < n * 9 / 2; f += kLinks) {
        const double2 p = u[2 * f], q = u[2 * f + 1];
        g32[out * 9 / 2 + f] = make_float4((float)p.x, (float)p.y, (float)q.x, (float)q.y);
    }
    for (int f = tid; f < n * 9 / 4; f += kLinks) {
        unsigned w[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const __half2 h = __halves2half2(__double2half(u[4 * f + k].x), __double2half(u[4 * f + k].y));
            w[k] = *reinterpret_cast<const unsigned *>(&h);
        }
        g16[out * 9 / 4 + f] = make_uint4(w[0], w[1], w[2], w[3]);
    }
}

// ------------------------------------------------------------------- source
// The two nonzero slices of P^dag (0, ..., 0, b4) as FP64 or block fields of two
// slices: P_+ b4 and P_- b4.  Thread per (lexicographic site, slice).
__global__ void __launch_bounds__(128) walls_kernel(const double *b4, FieldRef even, FieldRef odd, const int *eo2lex, int V)
{
    const size_t f = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
    if (f >= (size_t)2 * V) return;
    const int lex = (int)(f >> 1), w = (int)(f & 1), i = lex >> 1;
    const double *c = b4 + (size_t)lex * 24;
    double2 v[12];
#pragma unroll
    for (int p = 0; p < 12; ++p)   // pair p: spins 0, 1 (p even, P_+) or 2, 3
        v[p] = (p & 1) == w ? make_double2(c[canon_of_internal(2 * p)], c[canon_of_internal(2 * p + 1)])
                            : make_double2(0.0, 0.0);
    const FieldRef &half = lex == eo2lex[i] ? even : odd;
    if (half.fx) {
        longlong2 t[12];
        int e = fx_pack(v, FX_BITS, t);
        if (!fx_is_raw(e)) {   // the empty half takes the other's exponent: only the hop reads these blocks
            const int top = max(fx_half<0>(e), fx_half<1>(e));
            e = fx_word(top, top);
        }
        fx_st(half, i, w, 2, t, e);
    } else {
        st_pairs<DWF_F64>(half, i, w, 2, v);
    }
}

// The 5D source from the walls' hops h (FP64 fields of two slices, c / 2 applied):
// slice 0 = y0 P_+ b4 + h_0, slice Ls - 1 = y1 P_- b4 + h_1, zero between.
// Canonical: thread per 16 bytes of a wall (the rest is cleared by a memset).
__global__ void source_canon_kernel(const double *b4, FieldRef he, FieldRef ho, const int *eo2lex, double2 y, double *b5,
                                    int V, int Ls)
{
    const size_t f = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
    if (f >= (size_t)V * 24) return;
    const int w = f >= (size_t)V * 12;
    const size_t r = f - (w ? (size_t)V * 12 : 0);
    const int lex = (int)(r / 12), k = (int)(r - (size_t)lex * 12), spin = k / 3, a = k - spin * 3, i = lex >> 1;
    const double *h = reinterpret_cast<const double *>((lex == __ldg(eo2lex + i) ? he : ho).v);
    // the reals (re, im) of (spin, a): groups 2 a and 2 a + 1, pair spin >> 1 of the group
    const size_t at = (((size_t)i * 12 + 4 * a + (spin >> 1)) * 2 + w) * 2 + (spin & 1);
    double2 q = h ? make_double2(h[at], h[at + 8]) : make_double2(0.0, 0.0);
    if ((spin >> 1) == w) {
        const double2 b = __ldg(reinterpret_cast<const double2 *>(b4) + r);
        const double yw = w ? y.y : y.x;
        q = make_double2(yw * b.x + q.x, yw * b.y + q.y);
    }
    reinterpret_cast<double2 *>(b5)[((size_t)(w ? Ls - 1 : 0) * V) * 12 + r] = q;
}
// Internal half field f of parity par: thread per 16 bytes.
__global__ void source_half_kernel(const double *b4, FieldRef hf, const int *eo2lex, double2 y, double2 *f, int Vh, int Ls)
{
    const size_t n = (size_t)Vh * 12 * Ls;
    for (size_t j = blockIdx.x * (size_t)blockDim.x + threadIdx.x; j < n; j += (size_t)gridDim.x * blockDim.x) {
        const size_t row = j / Ls, i = row / 12;
        const int s = (int)(j - row * Ls), p = (int)(row - i * 12);
        double2 q = make_double2(0.0, 0.0);
        if (s == 0 || s == Ls - 1) {
            const int w = s ? 1 : 0;
            if (hf.v) q = reinterpret_cast<const double2 *>(hf.v)[row * 2 + w];
            if ((p & 1) == w) {
                const double *c = b4 + (size_t)__ldg(eo2lex + i) * 24;
                const double yw = w ? y.y : y.x;
                q = make_double2(yw * c[canon_of_internal(2 * p)] + q.x, yw * c[canon_of_internal(2 * p + 1)] + q.y);
            }
        }
        f[j] = q;
    }
}

}  // namespace

cudaError_t launch_pack_full(int prec, const double *canon, FieldRef even, FieldRef odd, const int *eo2lex, int Vh,
                             int V, int Ls, cudaStream_t st)
{
    (void)Vh;
    return launch_pack<true, false>(prec, canon, even, odd, eo2lex, V, Ls, st);
}

cudaError_t launch_unpack_full(int prec, FieldRef even, FieldRef odd, double *canon, const int *eo2lex, int Vh,
                               int V, int Ls, cudaStream_t st)
{
    (void)Vh;
    return launch_pack<true, true>(prec, canon, even, odd, eo2lex, V, Ls, st);
}

cudaError_t launch_pack_eo(int prec, const double *canon, FieldRef f, int Vh, int Ls, cudaStream_t st)
{
    return launch_pack<false, false>(prec, canon, f, f, nullptr, Vh, Ls, st);
}

cudaError_t launch_unpack_eo(int prec, FieldRef f, double *canon, int Vh, int Ls, cudaStream_t st)
{
    return launch_pack<false, true>(prec, canon, f, f, nullptr, Vh, Ls, st);
}

cudaError_t launch_pack_mix(int prec, const double *canon, FieldRef x, const MixArgs &a, cudaStream_t st)
{
    switch (prec) {
    case DWF_F64: return launch_pack_mix_p<DWF_F64>(canon, x, a, st);
    case DWF_F32: return launch_pack_mix_p<DWF_F32>(canon, x, a, st);
    case DWF_F16: return launch_pack_mix_p<DWF_F16>(canon, x, a, st);
    }
    return cudaErrorInvalidValue;
}

cudaError_t launch_links_to_limbs(const void *g64, int4 *gfx, int *ge, size_t n, cudaStream_t st)
{
    const size_t b = (n + 127) / 128;
    links_to_limbs_kernel<<<(unsigned)(b < 152 * 64 ? b : 152 * 64), 128, 0, st>>>((const double2 *)g64, gfx, ge, n);
    return cudaGetLastError();
}

cudaError_t launch_pack_gauge(const double *U, const int dims[4], const int bc[4], void *g64, void *g32, void *g16,
                              int4 *gfx, int *ge, cudaStream_t st)
{
    Dims D;
    for (int k = 0; k < 4; ++k) D.d[k] = dims[k], D.bc[k] = bc[k];
    const int Vh = dims[0] * dims[1] * dims[2] * dims[3] / 2;
    const unsigned g = (unsigned)(2 * (((long long)Vh * 8 + kLinks - 1) / kLinks));
    pack_gauge_kernel<<<g, kLinks, 0, st>>>(U, D, Vh, (double2 *)g64, (float4 *)g32, (uint4 *)g16, gfx, ge);
    return cudaGetLastError();
}

cudaError_t launch_walls(const double *b4, FieldRef even, FieldRef odd, const int *eo2lex, int V, cudaStream_t st)
{
    walls_kernel<<<(unsigned)(((size_t)2 * V + 127) / 128), 128, 0, st>>>(b4, even, odd, eo2lex, V);
    return cudaGetLastError();
}

cudaError_t launch_source_canon(const double *b4, FieldRef he, FieldRef ho, const int *eo2lex, double y0, double y1,
                                double *b5, int V, int Ls, cudaStream_t st)
{
    const size_t slice = (size_t)V * 24;
    if (Ls > 2) {
        const cudaError_t e = cudaMemsetAsync(b5 + slice, 0, (size_t)(Ls - 2) * slice * sizeof(double), st);
        if (e != cudaSuccess) return e;
    }
    source_canon_kernel<<<(unsigned)((slice + 255) / 256), 256, 0, st>>>(b4, he, ho, eo2lex, make_double2(y0, y1), b5, V, Ls);
    return cudaGetLastError();
}

cudaError_t launch_source_half(const double *b4, FieldRef hf, const int *eo2lex, double y0, double y1, FieldRef f, int Vh,
                               int Ls, cudaStream_t st)
{
    const size_t blocks = ((size_t)Vh * 12 * Ls + 255) / 256;
    source_half_kernel<<<(unsigned)(blocks < 152 * 64 ? blocks : 152 * 64), 256, 0, st>>>(
        b4, hf, eo2lex, make_double2(y0, y1), (double2 *)f.v, Vh, Ls);
    return cudaGetLastError();
}

}  // namespace dwf
