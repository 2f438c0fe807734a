// Site-local FP64 kernels on fixed-point blocks (fixed.cuh): fifth-direction
// mixing, the CG direction update and the conversion of FP64 fields to blocks.
#include "fx_fields.cuh"

namespace dwf {
namespace {

struct TileSmem {
    int4 *tile;   // [SB][fx_site_stride(Ls)]
    int *te;      // [SB][Ls]
};
__device__ __forceinline__ TileSmem tile_smem_fx(unsigned char *raw, int Ls, int SB)
{
    TileSmem t;
    t.tile = reinterpret_cast<int4 *>(raw);
    t.te = reinterpret_cast<int *>(t.tile + SB * fx_site_stride(Ls));
    return t;
}
size_t tile_bytes_fx(int Ls, int SB) { return (size_t)SB * (fx_site_stride(Ls) * sizeof(int4) + Ls * sizeof(int)); }

// out(site, s) = sum_t M[chi][s][t] in(site, t); FP64 or block fields
__global__ void __launch_bounds__(128) mix_fx_kernel(const MixArgs a)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int Ls = a.Ls, s = threadIdx.x, j = threadIdx.y, B = fx_mix_bits(Ls);
    const int site = blockIdx.x * blockDim.y + j;
    const bool active = site < a.Vh;
    const TileSmem sm = tile_smem_fx(smem_raw, Ls, blockDim.y);
    int4 *tile = sm.tile + j * fx_site_stride(Ls);
    int *te = sm.te + j * Ls;
    if (active) {
        longlong2 t[12];
        int e;
        if (a.in.fx) {
            fx_ld<true>(a.in, (size_t)site, s, Ls, t);
            e = a.in.fx[(size_t)site * Ls + s];
            if (!fx_is_raw(e))
#pragma unroll
                for (int k = 0; k < 12; ++k) t[k] = make_longlong2(t[k].x >> (FX_BITS - B), t[k].y >> (FX_BITS - B));
        } else {
            double2 v[12];
            ld_pairs<DWF_F64, true>(a.in, (size_t)site, s, Ls, v);
            e = fx_pack(v, B, t);
        }
        fx_put(tile + s * FX_ROW, t, e);
        te[s] = e;
    }
    __syncthreads();
    if (active) {
        FxSum S;
        fx_mix(FxMat{a.mat_fx, reinterpret_cast<const double *>(a.mat), a.band}, tile, te, s, Ls, B, S);
        fx_store_sum(a.out, (size_t)site, s, Ls, S, B);
    }
}

// x += alpha p (deferred, see CgUpdateArgs); p = r + beta p (or p = r); phat = M p as blocks
__global__ void __launch_bounds__(128) cg_update_fx_kernel(const CgUpdateArgs a)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int Ls = a.Ls, s = threadIdx.x, j = threadIdx.y, B = fx_mix_bits(Ls);
    const int site = blockIdx.x * blockDim.y + j;
    const bool active = site < a.Vh;
    const TileSmem sm = tile_smem_fx(smem_raw, Ls, blockDim.y);
    int4 *tile = sm.tile + j * fx_site_stride(Ls);
    int *te = sm.te + j * Ls;
    if (active) {
        double2 r[12], p[12];
        ld_pairs<DWF_F64, false>(a.r, (size_t)site, s, Ls, r);
        const double xal = a.xacc ? a.scal->alpha : 0.0;
        if (!a.init || xal != 0.0) ld_pairs<DWF_F64, false>(a.p, (size_t)site, s, Ls, p);
        if (xal != 0.0) {
            FieldRef xf;
            xf.v = a.xacc;
            double2 xv[12];
            ld_pairs<DWF_F64, false>(xf, (size_t)site, s, Ls, xv);
#pragma unroll
            for (int k = 0; k < 12; ++k) xv[k] = p_fma(p_splat(xal), p[k], xv[k]);
            st_pairs<DWF_F64>(xf, (size_t)site, s, Ls, xv);
        }
        if (a.init) {
#pragma unroll
            for (int k = 0; k < 12; ++k) p[k] = r[k];
        } else {
            const double2 be = p_splat(a.scal->beta);
#pragma unroll
            for (int k = 0; k < 12; ++k) p[k] = p_fma(be, p[k], r[k]);
        }
        st_pairs<DWF_F64>(a.p, (size_t)site, s, Ls, p);
        longlong2 t[12];
        const int e = fx_pack(p, B, t);
        fx_put(tile + s * FX_ROW, t, e);
        te[s] = e;
    }
    __syncthreads();
    if (active) {
        FxSum S;
        fx_mix(FxMat{a.mat_fx, reinterpret_cast<const double *>(a.mat), a.band}, tile, te, s, Ls, B, S);
        fx_store_sum(a.phat, (size_t)site, s, Ls, S, B);
    }
}

__global__ void __launch_bounds__(128) to_blocks_kernel(FieldRef in, FieldRef out, size_t n, int Ls)
{
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
        const size_t site = i / Ls;
        const int s = (int)(i - site * Ls);
        double2 v[12];
        longlong2 t[12];
        ld_pairs<DWF_F64, true>(in, site, s, Ls, v);
        const int e = fx_pack(v, FX_BITS, t);
        fx_st(out, site, s, Ls, t, e);
    }
}

}  // namespace

size_t exponent_bytes(int Vh, int Ls) { return (size_t)Vh * Ls * sizeof(int); }

cudaError_t launch_mix_fx(const MixArgs &a, cudaStream_t st)
{
    static unsigned long long optin = 0;
    cudaError_t e = smem_optin(mix_fx_kernel, 200 * 1024, optin);
    if (e != cudaSuccess) return e;
    const int SB = 128 / a.Ls;
    mix_fx_kernel<<<(a.Vh + SB - 1) / SB, dim3(a.Ls, SB), tile_bytes_fx(a.Ls, SB), st>>>(a);
    return cudaGetLastError();
}

cudaError_t launch_cg_update_fx(const CgUpdateArgs &a, cudaStream_t st)
{
    static unsigned long long optin = 0;
    cudaError_t e = smem_optin(cg_update_fx_kernel, 200 * 1024, optin);
    if (e != cudaSuccess) return e;
    const int SB = 128 / a.Ls;
    cg_update_fx_kernel<<<(a.Vh + SB - 1) / SB, dim3(a.Ls, SB), tile_bytes_fx(a.Ls, SB), st>>>(a);
    return cudaGetLastError();
}

cudaError_t launch_to_blocks(FieldRef in, FieldRef out, int rows, int Ls, cudaStream_t st)
{
    const size_t n = (size_t)rows * Ls, blocks = (n + 127) / 128;
    to_blocks_kernel<<<(unsigned)(blocks > 152 * 64 ? 152 * 64 : blocks), 128, 0, st>>>(in, out, n, Ls);
    return cudaGetLastError();
}

}  // namespace dwf
