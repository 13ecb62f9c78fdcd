// adjoint_tiles.cu -- the adjoint of the deposit: per-particle setup, launch of
// the (tile, particle) sums (adjoint_kernel.cuh), and the chain rule.
#include "adjoint_kernel.cuh"
#include "twosum.cuh"

namespace rubix {

// ---------------------------------------------------------------------------
// Setup: each sorted particle's position (ta, tz) in its SSP cell.
// ---------------------------------------------------------------------------
__global__ void k_adj_setup(const AdjointParams P, float2* __restrict__ wu) {
    const long long n_in = P.seg_off[(long long)P.n_s * P.n_bands];
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n_in;
         i += (long long)gridDim.x * blockDim.x) {
        const PartRec pr = P.prec[i];
        int ia, iz;
        float ta, tz, dta, dtz;
        ssp_cell(log10f(pr.age), P.ssp.la_nodes, P.ssp.n_age, ia, ta, dta);
        ssp_cell(log10f(pr.Z), P.ssp.lz_nodes, P.ssp.n_Z, iz, tz, dtz);
        wu[i] = make_float2(ta, tz);
    }
}

int launch_adjoint_setup(const AdjointParams& P, float2* wu, cudaStream_t st) {
    if (P.n_in <= 0) return 0;
    long long nb = (P.n_in + 255) / 256;
    if (nb > 16ll * sm_count()) nb = 16ll * sm_count();
    k_adj_setup<<<(int)nb, 256, 0, st>>>(P, wu);
    return 1;
}

int launch_adjoint_tiles(const AdjTileParams& P, int n_ctas, int threads, size_t smem, cudaStream_t st) {
    const int B = kind_bins(P.kind);
    if (P.tile_w % B != 0) return -1;
    const int R = P.tile_w / B;
    const bool mean = P.resample != 0;
    const AdjointFn fn = P.kind == 0 ? adjoint_fn_k0(R, mean)
                                     : (P.kind == 1 ? adjoint_fn_k1(R, mean) : adjoint_fn_k2(R, mean));
    if (!fn) return -1;
    if (cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess) return -1;
    fn<<<n_ctas, threads, smem, st>>>(P);
    return 1;
}

// ---------------------------------------------------------------------------
// K8: tiles summed in tile order (compensated FP32), chain rule, original order.
// ---------------------------------------------------------------------------
__global__ void k_adj_final(const AdjointParams P, const float4* __restrict__ part, int n_tiles, long long n_cap) {
    const long long n_in = P.seg_off[(long long)P.n_s * P.n_bands];
    const float ln10 = 2.302585092994046f;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n_in;
         i += (long long)gridDim.x * blockDim.x) {
        // the tiles' sums in tile order, compensated (two-sum) in FP32
        float sm = 0.f, sa = 0.f, sz = 0.f, sv = 0.f, em = 0.f, ea = 0.f, ez = 0.f, ev = 0.f;
        for (int t = 0; t < n_tiles; ++t) {
            const float4 v = part[t * n_cap + i];
            two_sum_add(sm, em, v.x);
            two_sum_add(sa, ea, v.y);
            two_sum_add(sz, ez, v.z);
            two_sum_add(sv, ev, v.w);
        }
        sm += em;
        sa += ea;
        sz += ez;
        sv += ev;
        const PartRec pr = P.prec[i];
        int ia, iz;
        float ta, tz, dta, dtz;
        ssp_cell(log10f(pr.age), P.ssp.la_nodes, P.ssp.n_age, ia, ta, dta);
        ssp_cell(log10f(pr.Z), P.ssp.lz_nodes, P.ssp.n_Z, iz, tz, dtz);
        // dt/dv = -(t + ls0/dls) / (c (1 + v/c)): the sums carry the (t + ls0/dls) factor
        const float q = -1.f / ((float)kC_kms + pr.v);  // = -1 / (c (1 + v/c))
        const float fs = (float)P.flux_scale;
        const float dm = fs * sm;
        const float dage = fs * pr.mass * dta * sa / (pr.age * ln10);
        const float dZ = fs * pr.mass * dtz * sz / (pr.Z * ln10);
        const float dv = fs * pr.mass * q * sv;
        const int p = P.perm[i];
        if (P.d_mass) P.d_mass[p] = dm;
        if (P.d_age) P.d_age[p] = dage;
        if (P.d_Z) P.d_Z[p] = dZ;
        if (P.d_v) P.d_v[p] = dv;
        if (P.contrib) {
            const float2 da = P.dv_dang ? P.dv_dang[p] : make_float2(0.f, 0.f);
            P.contrib[kGlobal * i] = (double)dv;
            P.contrib[kGlobal * i + 1] = (double)pr.mass * (double)dm;
            P.contrib[kGlobal * i + 2] = (double)dv * (double)da.x;
            P.contrib[kGlobal * i + 3] = (double)dv * (double)da.y;
        }
    }
}

int launch_adjoint_final(const AdjointParams& P, const float4* part, int n_tiles, long long n_cap, cudaStream_t st) {
    if (P.n_in <= 0) return 0;
    long long nb = (P.n_in + 255) / 256;
    if (nb > 16ll * sm_count()) nb = 16ll * sm_count();
    k_adj_final<<<(int)nb, 256, 0, st>>>(P, part, n_tiles, n_cap);
    return 1;
}

}  // namespace rubix
