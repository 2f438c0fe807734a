// The FP64 hop on block fixed-point fields (fixed.cuh): the default of the FP64
// operator.  Same launch, arguments and epilogue as the hop of hop_kernels.cuh;
// the input field is a block field, y and the output FP64 or block fields, rin FP64.
//
// A CTA takes SB sites x all Ls slices, one (site, s) per thread.  Its sites' links
// come to shared memory as limbs, made when the links are set (turning FP64 links into
// limbs here cost 2 % at Ls 16, 8 % at Ls 10 and half of the two-slice source: 1632
// against 725 us at 24^3x48).  The threads walk the eight directions in one loop (unrolled, its code
// no longer fits the instruction cache): each has its neighbour's block copied
// asynchronously into its own shared slots one direction ahead, projects, multiplies
// and reconstructs in integers.  The eight directions' exponents are known before
// the first product (the larger half's + link exponent), so all are summed against the
// largest.
//
// Bound: the multiply pipe, 216 multiply-adds of four cycles per direction and warp,
// closely followed by the integer adds and shifts (342 of two cycles) and the issue
// slots; DRAM is 15 % busy.  At 16^3x32, Ls 16 (K_a, dense mixing): 498 us against
// 1987 us on the FP64 pipe (485 us with one exponent for both halves of a block).  In
// an earlier form of 502 us (links made into limbs here) the eight directions took
// about 267 us and the mixing about 155 us, bound by its shared-memory reads.  All
// forms use 128 registers; their spills (250 to 490 bytes a thread) lie on paths that are
// seldom taken: 0.2 % of the executed instructions access local memory.
#pragma once

#include "fx_fields.cuh"   // before stencil.cuh: its templates take the integer pairs
#include "stencil.cuh"

namespace dwf {
namespace {

// Q = U H >> sh for a half spinor of integers below 2^60: u nine complex entries
// below 2^59 as limbs {re low, re high, im low, im high} of radix 2^31.  In units of
// 2^(e - 59) for H and 2^(eu - 59) for U, Q comes in 2^(e + eu - 56); the sums of the
// cross products stay below 2^62.6 and are rounded at 2^31, eight directions' Q below
// 2^62.6.
template <bool GLOBAL>
__device__ __forceinline__ void fx_su3(const int4 *u, const longlong2 *Hx, const longlong2 *Hy, int sh, longlong2 *Qx,
                                       longlong2 *Qy)
{
    int32_t xl[3][2], xh[3][2], yl[3][2], yh[3][2];
#pragma unroll
    for (int b = 0; b < 3; ++b) {
        fx_limbs31(Hx[b].x, xl[b][0], xh[b][0]);
        fx_limbs31(Hx[b].y, xl[b][1], xh[b][1]);
        fx_limbs31(Hy[b].x, yl[b][0], yh[b][0]);
        fx_limbs31(Hy[b].y, yl[b][1], yh[b][1]);
    }
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        int64_t rh[2], rx[2], ih[2], ix[2];
#pragma unroll
        for (int p = 0; p < 2; ++p) rh[p] = ih[p] = 0, rx[p] = ix[p] = 1 << 30;
#pragma unroll
        for (int b = 0; b < 3; ++b) {
            const int4 q = GLOBAL ? __ldg(u + a * 3 + b) : u[a * 3 + b];
#pragma unroll
            for (int p = 0; p < 2; ++p) {
                fx_mad(xl[b][p], xh[b][p], q.x, q.y, rh[p], rx[p]);
                fx_mad(yl[b][p], yh[b][p], -q.z, -q.w, rh[p], rx[p]);
                fx_mad(yl[b][p], yh[b][p], q.x, q.y, ih[p], ix[p]);
                fx_mad(xl[b][p], xh[b][p], q.z, q.w, ih[p], ix[p]);
            }
        }
        Qx[a] = make_longlong2((rh[0] + (rx[0] >> 31)) >> sh, (rh[1] + (rx[1] >> 31)) >> sh);
        Qy[a] = make_longlong2((ih[0] + (ix[0] >> 31)) >> sh, (ih[1] + (ix[1] >> 31)) >> sh);
    }
}

// direction d's half spinor from a block, and its product into the sum
template <bool DAG>
__device__ __forceinline__ void fx_project(int d, const longlong2 *v, longlong2 *Hx, longlong2 *Hy)
{
    constexpr int F = DAG ? -1 : 1;
    switch (d) {
    case 0: project<0, F>(v, Hx, Hy); break;
    case 1: project<1, F>(v, Hx, Hy); break;
    case 2: project<2, F>(v, Hx, Hy); break;
    case 3: project<3, F>(v, Hx, Hy); break;
    case 4: project<0, -F>(v, Hx, Hy); break;
    case 5: project<1, -F>(v, Hx, Hy); break;
    case 6: project<2, -F>(v, Hx, Hy); break;
    default: project<3, -F>(v, Hx, Hy); break;
    }
}
template <bool DAG>
__device__ __forceinline__ void fx_reconstruct(int d, longlong2 *acc, const longlong2 *Qx, const longlong2 *Qy)
{
    constexpr int F = DAG ? -1 : 1;
    switch (d) {
    case 0: reconstruct<0, F>(acc, Qx, Qy); break;
    case 1: reconstruct<1, F>(acc, Qx, Qy); break;
    case 2: reconstruct<2, F>(acc, Qx, Qy); break;
    case 3: reconstruct<3, F>(acc, Qx, Qy); break;
    case 4: reconstruct<0, -F>(acc, Qx, Qy); break;
    case 5: reconstruct<1, -F>(acc, Qx, Qy); break;
    case 6: reconstruct<2, -F>(acc, Qx, Qy); break;
    default: reconstruct<3, -F>(acc, Qx, Qy); break;
    }
}

// one thread's block of a neighbour, 12 asynchronous 16-byte copies into its own
// slots (vector k of thread tid at [k nt + tid])
__device__ __forceinline__ void fx_fetch(int4 *slot, int nt, const FieldRef &in, int nb, int s, int Ls)
{
    const longlong2 *p = reinterpret_cast<const longlong2 *>(in.v) + ((size_t)nb * 12) * Ls + s;
    const uint32_t d = (uint32_t)__cvta_generic_to_shared(slot);
#pragma unroll
    for (int k = 0; k < 12; ++k)
        asm volatile("cp.async.ca.shared.global [%0], [%1], 16;" ::"r"(d + k * nt * 16), "l"(p + (size_t)k * Ls) : "memory");
    asm volatile("cp.async.commit_group;" ::: "memory");
}

// the half of a block in its slots that lies lower, by |above| bits, shifted to the
// other's exponent; out of line, as fields seldom need it (fx_near)
__device__ __noinline__ void fx_even_halves(int4 *slot, int nt, int above)
{
    const int c = above > 0, sh = above > 0 ? above : -above;
    for (int k = c; k < 12; k += 2) {
        longlong2 *q = reinterpret_cast<longlong2 *>(slot + k * nt);
        *q = make_longlong2(q->x >> sh, q->y >> sh);
    }
}

// one direction in FP64, for sites with non-finite neighbours or links
template <bool DAG, int D>
__device__ __forceinline__ void fx_dir_double(double2 *acc, const FieldRef &in, int nb, int s, int Ls, const double *U)
{
    constexpr int MU = D & 3;
    constexpr int SIG = (D < 4 ? 1 : -1) * (DAG ? -1 : 1);
    double2 v[12], u[9];
    load_link<DWF_F64, true>(U + D * 18, u);
    fx_ld_double<true>(in, (size_t)nb, s, Ls, v);
    hop_one<MU, SIG>(acc, u, v);
}
template <bool DAG>
__device__ __noinline__ void fx_hop_raw(FieldRef in, const int *nb, const double *U, int s, int Ls, double2 *acc)
{
#pragma unroll
    for (int k = 0; k < 12; ++k) acc[k] = make_double2(0.0, 0.0);
    fx_dir_double<DAG, 0>(acc, in, nb[0], s, Ls, U);
    fx_dir_double<DAG, 1>(acc, in, nb[1], s, Ls, U);
    fx_dir_double<DAG, 2>(acc, in, nb[2], s, Ls, U);
    fx_dir_double<DAG, 3>(acc, in, nb[3], s, Ls, U);
    fx_dir_double<DAG, 4>(acc, in, nb[4], s, Ls, U);
    fx_dir_double<DAG, 5>(acc, in, nb[5], s, Ls, U);
    fx_dir_double<DAG, 6>(acc, in, nb[6], s, Ls, U);
    fx_dir_double<DAG, 7>(acc, in, nb[7], s, Ls, U);
}

// shared memory of one CTA: links as limbs, the tile (before it is filled: the
// neighbour blocks in flight, 12 vectors per thread), exponents of links and rows
struct FxSmem {
    int4 *u;      // [SB][8][9]
    int4 *tile;   // [SB][fx_site_stride(Ls)]
    int *eu;      // [SB][8]
    int *nb;      // [SB][8] neighbours
    int *te;      // [SB][Ls]
};
// two slices (the 5D source) read their links from global memory: with two threads to
// a site, staging them would only cost occupancy
__host__ __device__ constexpr bool fx_global_links(int Ls) { return Ls == 2; }
__host__ __device__ inline size_t fx_smem_bytes(int Ls, int SB)
{
    return (size_t)SB * ((fx_global_links(Ls) ? 0 : 72) + fx_site_stride(Ls)) * sizeof(int4) +
           (size_t)SB * (16 + Ls) * sizeof(int);
}

// LS: Ls, or 0 for any (the fixed ones save the address arithmetic)
template <bool DAG, int LS>
__global__ void __launch_bounds__(128, 4) hop_fx_kernel(const HopArgs a)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int Ls = LS ? LS : a.Ls, SB = LS ? 128 / LS : (int)blockDim.y, s = threadIdx.x, j = threadIdx.y;
    const int tid = j * Ls + s, nt = Ls * SB, B = fx_mix_bits(Ls);
    // in a sweep every CTA is full (hop_fx_launch_ls); the two-slice source has none
    const int site0 = LS == 2 ? blockIdx.x * SB : sweep_site(a, blockIdx.x * SB), site = site0 + j;
    const bool active = site < a.Vh;
    FxSmem sm;
    constexpr bool GL = fx_global_links(LS);
    sm.u = reinterpret_cast<int4 *>(smem_raw);
    sm.tile = sm.u + (GL ? 0 : SB * 72);
    sm.eu = reinterpret_cast<int *>(sm.tile + SB * fx_site_stride(Ls));
    sm.nb = sm.eu + SB * 8;
    sm.te = sm.nb + SB * 8;
    int4 *tile = sm.tile + j * fx_site_stride(Ls), *row = tile + s * FX_ROW, *slot = sm.tile + tid;
    int *te = sm.te + j * Ls;
    const int *nb = sm.nb + j * 8;

    const int nsites = min(SB, a.Vh - site0);
    if (!GL) {
        const int4 *src = a.gauge_fx + (size_t)site0 * 72;
        const uint32_t d = (uint32_t)__cvta_generic_to_shared(sm.u);
        for (int i = tid; i < nsites * 72; i += nt)
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d + i * 16), "l"(src + i) : "memory");
        asm volatile("cp.async.commit_group;" ::: "memory");
    }
    for (int i = tid; i < nsites * 8; i += nt) {
        sm.nb[i] = __ldg(a.nbr + (size_t)site0 * 8 + i);
        sm.eu[i] = __ldg(a.gauge_e + (size_t)site0 * 8 + i);
    }
    int e8[8];
    if (active) {
        const int4 *p = reinterpret_cast<const int4 *>(a.nbr + (size_t)site * 8);
        const int4 q0 = __ldg(p), q1 = __ldg(p + 1);
        fx_fetch(slot, nt, a.in, q0.x, s, Ls);
        const int n8[8] = {q0.x, q0.y, q0.z, q0.w, q1.x, q1.y, q1.z, q1.w};
#pragma unroll
        for (int d = 0; d < 8; ++d) e8[d] = __ldg(a.in.fx + (size_t)n8[d] * Ls + s);
    } else {
        asm volatile("cp.async.commit_group;" ::: "memory");   // the same number of groups as the others
    }
    asm volatile("cp.async.wait_group 1;" ::: "memory");   // the links; the first block may still be on its way
    __syncthreads();

    longlong2 acc[12];
    int emax = 2 * FX_ZERO;
    bool raw = false;
#pragma unroll
    for (int k = 0; k < 12; ++k) acc[k] = make_longlong2(0, 0);
    if (active) {
        uint64_t shifts = 0, above = 0;   // eight bits per direction: emax - e, at most 63, and how far P_+ lies above P_-
        bool uneven = false;
#pragma unroll
        for (int d = 0; d < 8; ++d) {
            const int eu = sm.eu[j * 8 + d], ep = fx_half<0>(e8[d]), em = fx_half<1>(e8[d]);
            raw = raw || fx_is_raw(e8[d]) || eu == FX_RAW;
            uneven = uneven || ep != em;
            e8[d] = max(ep, em) + eu;
            emax = max(emax, e8[d]);
        }
#pragma unroll
        for (int d = 0; d < 8; ++d) shifts |= (uint64_t)(uint32_t)min(emax - e8[d], 63) << (8 * d);
        if (uneven) {   // rare in fields (fx_near): projecting takes both halves at the larger exponent
#pragma unroll 1
            for (int d = 0; d < 8; ++d) {
                const int e = __ldg(a.in.fx + (size_t)nb[d] * Ls + s), ep = fx_half<0>(e), em = fx_half<1>(e);
                const int ab = ep == FX_ZERO || em == FX_ZERO ? 0 : min(max(ep - em, -63), 63);   // zeros need no shift
                above |= (uint64_t)(uint32_t)(ab & 0xff) << (8 * d);
            }
        }
        const int4 *u = GL ? a.gauge_fx + (size_t)site * 72 : sm.u + j * 72;
#pragma unroll 1
        for (int d = 0; d < 8; ++d) {
            longlong2 Hx[3], Hy[3], Qx[3], Qy[3];
            asm volatile("cp.async.wait_group 0;" ::: "memory");
            if (above) fx_even_halves(slot, nt, (int8_t)(above >> (8 * d)));
            {
                longlong2 v[12];
#pragma unroll
                for (int k = 0; k < 12; ++k) v[k] = *reinterpret_cast<const longlong2 *>(slot + k * nt);
                fx_project<DAG>(d, v, Hx, Hy);
            }
            if (d < 7) fx_fetch(slot, nt, a.in, nb[d + 1], s, Ls);   // into the same slots: this block is in registers
            fx_su3<GL>(u + d * 9, Hx, Hy, (int)(shifts >> (8 * d)) & 63, Qx, Qy);
            fx_reconstruct<DAG>(d, acc, Qx, Qy);
        }
    }
    __syncthreads();   // the slots become the tile
    if (active) {
        if (raw) {
            double2 o[12];
            fx_hop_raw<DAG>(a.in, a.nbr + (size_t)site * 8,
                            reinterpret_cast<const double *>(a.gauge) + (size_t)site * 8 * 18, s, Ls, o);
            const int e = fx_pack(o, B, acc);
            fx_put(row, acc, e);
            te[s] = e;
        } else {
            const int wp = fx_half_width<0>(acc), wm = fx_half_width<1>(acc);
            te[s] = fx_word(fx_half_zero<0>(acc) ? FX_ZERO : emax - 56 + wp, fx_half_zero<1>(acc) ? FX_ZERO : emax - 56 + wm);
#pragma unroll
            for (int k = 0; k < 12; ++k)
                acc[k] = make_longlong2(fx_align(acc[k].x, k & 1 ? wm : wp, 63 - B), fx_align(acc[k].y, k & 1 ? wm : wp, 63 - B));
            fx_put(row, acc, 0);
        }
    }
    __syncthreads();

    FxSum S;
    if (active) fx_mix(FxMat{a.post_fx, reinterpret_cast<const double *>(a.post), a.post_band}, tile, te, s, Ls, B, S);
    if (a.ymode == 2) {
        __syncthreads();
        if (active) {
            longlong2 t[12];
            int e;
            if (a.y.fx) {
                fx_ld<false>(a.y, (size_t)site, s, Ls, t);
                e = a.y.fx[(size_t)site * Ls + s];
                if (!fx_is_raw(e))
#pragma unroll
                    for (int k = 0; k < 12; ++k) t[k] = make_longlong2(t[k].x >> (FX_BITS - B), t[k].y >> (FX_BITS - B));
            } else {
                double2 y[12];
                ld_pairs<DWF_F64, false>(a.y, (size_t)site, s, Ls, y);
                e = fx_pack(y, B, t);
            }
            fx_put(row, t, e);
            te[s] = e;
        }
        __syncthreads();
        if (active) {
            FxSum T;
            fx_mix(FxMat{a.y_fx, reinterpret_cast<const double *>(a.ymat), a.y_band}, tile, te, s, Ls, B, T);
            fx_sum_add(S, T, B);
        }
    }
    if (a.ymode != 1 && !a.rin.v && !a.zmat && a.red.op == RED_NONE) {   // nothing left that works on doubles
        if (active) fx_store_sum(a.out, (size_t)site, s, Ls, S, B);
        return;
    }
    double2 o[12];
    double nrm = 0;
    if (active) {
        fx_sum_doubles(S, B, o);
        if (a.ymode == 1) {
            double2 y[12];
            fx_ld_double<false>(a.y, (size_t)site, s, Ls, y);
#pragma unroll
            for (int k = 0; k < 12; ++k) o[k] = p_add(o[k], y[k]);
        }
        if (a.rin.v) {
            const double nal = -*a.ralpha;
            double2 r[12];
            ld_pairs<DWF_F64, false>(a.rin, (size_t)site, s, Ls, r);
#pragma unroll
            for (int k = 0; k < 12; ++k) o[k] = p_fma(p_splat(nal), o[k], r[k]);
        }
        if (a.red.op != RED_NONE) {
            double2 s2 = make_double2(0.0, 0.0);
#pragma unroll
            for (int k = 0; k < 12; ++k) s2 = p_fma(o[k], o[k], s2);
            nrm = s2.x + s2.y;
        }
    }
    if (a.zmat) {
        __syncthreads();
        if (active) {
            longlong2 t[12];
            const int e = fx_pack(o, B, t);
            fx_put(row, t, e);
            te[s] = e;
        }
        __syncthreads();
        if (active) {
            fx_mix(FxMat{a.z_fx, reinterpret_cast<const double *>(a.zmat), a.z_band}, tile, te, s, Ls, B, S);
            fx_store_sum(a.out, (size_t)site, s, Ls, S, B);
        }
    } else if (active) {
        fx_store_double(a.out, (size_t)site, s, Ls, o);
    }
    if (a.red.op != RED_NONE) grid_reduce(nrm, a.red);
}

}  // namespace

template <bool DAG, int LS>
cudaError_t hop_fx_launch_ls(const HopArgs &a, cudaStream_t st)
{
    static unsigned long long optin = 0;
    cudaError_t e = smem_optin(hop_fx_kernel<DAG, LS>, 200 * 1024, optin);
    if (e != cudaSuccess) return e;
    const int SB = 128 / a.Ls;
    HopArgs b = a;
    if (b.zblock > 0 && (b.zblock * b.ext[0] * b.ext[1]) % SB) b.zblock = 0;   // a CTA would straddle two runs
    hop_fx_kernel<DAG, LS><<<(a.Vh + SB - 1) / SB, dim3(a.Ls, SB), fx_smem_bytes(a.Ls, SB), st>>>(b);
    return cudaGetLastError();
}

template <bool DAG>
cudaError_t hop_fx_launch(const HopArgs &a, cudaStream_t st)
{
    switch (a.Ls) {
    case 2: return hop_fx_launch_ls<DAG, 2>(a, st);
    case 8: return hop_fx_launch_ls<DAG, 8>(a, st);
    case 12: return hop_fx_launch_ls<DAG, 12>(a, st);
    case 16: return hop_fx_launch_ls<DAG, 16>(a, st);
    default: return hop_fx_launch_ls<DAG, 0>(a, st);
    }
}

}  // namespace dwf
