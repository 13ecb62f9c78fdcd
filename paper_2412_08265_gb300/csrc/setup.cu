// setup.cu -- K3 of the deposit path (Sec. 3: each star's SSP lookup and
// Doppler shift, prepared once per particle): every in-field particle, in
// sorted order, becomes a 32-byte record for the deposit (its four mass-scaled
// bilinear corner weights, its cell, its Doppler shift in fixed point, the rounds it
// takes) and a 16-byte one with the affine map t(j) = B + jA from output bin j to
// the fractional SSP node position, and each spaxel's particles are cut into work
// items of at most `chunk` particles.
#include "common.cuh"
#include "kernels.h"
#include "sort_layout.h"

namespace rubix {

// ----------------------------------------------------------------------------
// Double-float arithmetic: a value is an unevaluated sum hi + lo of two FP32
// numbers (|lo| <= ulp(hi) / 2), about 48 significant bits. Products use the
// exact FMA residual, sums Knuth's two-sum; each operation is a handful of
// FP32 instructions instead of one FP64 instruction on this GPU's FP64 pipe,
// which runs at 1/64 of the FP32 rate (Dekker 1971; Shewchuk 1997).
// ----------------------------------------------------------------------------
struct DF {
    float hi, lo;
};

// (the _rn intrinsics keep the compiler from contracting these products and
// sums into FMAs, which the error-free transformations must not see)
__device__ __forceinline__ DF df_norm(float hi, float lo) {  // |hi| >= |lo|
    const float s = __fadd_rn(hi, lo);
    return DF{s, __fsub_rn(lo, __fsub_rn(s, hi))};
}

__device__ __forceinline__ DF df_of(double x) {
    const float hi = (float)x;
    return DF{hi, (float)(x - (double)hi)};
}

__device__ __forceinline__ DF df_add(DF a, DF b) {
    const float s = __fadd_rn(a.hi, b.hi);
    const float z = __fsub_rn(s, a.hi);
    const float e = __fadd_rn(__fsub_rn(a.hi, __fsub_rn(s, z)), __fsub_rn(b.hi, z));
    return df_norm(s, __fadd_rn(e, __fadd_rn(a.lo, b.lo)));
}

__device__ __forceinline__ DF df_neg(DF a) { return DF{-a.hi, -a.lo}; }

__device__ __forceinline__ DF df_mul(DF a, DF b) {
    const float p = __fmul_rn(a.hi, b.hi);
    const float e = fmaf(a.hi, b.hi, -p);
    return df_norm(p, fmaf(a.hi, b.lo, fmaf(a.lo, b.hi, e)));
}

__device__ __forceinline__ DF df_mul_f(DF a, float b) {
    const float p = __fmul_rn(a.hi, b);
    const float e = fmaf(a.hi, b, -p);
    return df_norm(p, fmaf(a.lo, b, e));
}

// x * scale (a power of two) rounded to an integer; saturates.
__device__ __forceinline__ int df_fixed(DF x, float scale) {
    const float v = x.hi * scale;  // exact
    const int i = __float2int_rn(v);
    return i + __float2int_rn(__fadd_rn(v - (float)i, x.lo * scale));
}

// ----------------------------------------------------------------------------
// K3: per-particle setup (sorted order).
// ----------------------------------------------------------------------------
__global__ void k_setup(SetupParams P) {
    const long long n_in = P.seg_off[(long long)P.n_s * P.n_bands];
    if (n_in > P.n_cap) return;
    const int n_ls = P.ssp.n_ls;
    // t(j) = ((l0 + j dl) / dop - ls0) / dls = B + j A with dop = (1 + z)(1 + v/c).
    // With alpha_z = 1 / ((1 + z) dls) and g = (v/c) / (1 + v/c), so that
    // 1 / (1 + v/c) = 1 - g:
    //   A = A_z (1 - g),   A_z = dl alpha_z,
    //   B = B_z - L g,     L = l0 alpha_z,  B_z = L - ls0/dls,
    // (bin means: B - A/2, the bin's lower edge), the particle's part in
    // double-float from the FP64 constants below (converted once per thread).
    const DF Az = df_of(P.dl * P.alpha_z), L = df_of(P.l0 * P.alpha_z);
    const DF Bz = df_of(fma(P.l0, P.alpha_z, -P.ls0_dls)), invc = df_of(P.inv_c);
    // the shift s(j) = -g (L' + j A_z) of DepRec at j = jc, L' = L (bin centres)
    // or L - A_z / 2 (edges), and its step -g A_z
    const DF Ls = df_of(P.l0 * P.alpha_z + ((double)P.jc - (P.resample ? 0.5 : 0.0)) * (P.dl * P.alpha_z));
    const float sc = __int_as_float((127 + P.fb) << 23), scg = __int_as_float((127 + P.fb + 13) << 23);
    const int nzc = max(P.ssp.n_Z, 2);
    const float t_lastj = (float)(P.resample ? P.n_lambda : P.n_lambda - 1);
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n_in;
         i += (long long)gridDim.x * blockDim.x) {
        const PartRec pr = P.pin[P.perm[i]];
        const float m = pr.mass, age = pr.age, Z = pr.Z;
        int ia, iz;
        float ta, tz, dta, dtz;
        ssp_cell(log10f(age), P.ssp.la_nodes, P.ssp.n_age, ia, ta, dta);
        ssp_cell(log10f(Z), P.ssp.lz_nodes, P.ssp.n_Z, iz, tz, dtz);
        const float ms = (float)P.flux_scale * m;
        DepRec r;
        MapRec mr;
        r.w[0] = ms * ((1.f - ta) * (1.f - tz));
        r.w[1] = ms * (ta * (1.f - tz));
        r.w[2] = ms * ((1.f - ta) * tz);
        r.w[3] = ms * (ta * tz);
        const int c0 = ia * P.ssp.n_Z + iz;  // SSP cell: its first entry among the age pairs
        // b = v/c, q = 1 + b, g = b / q: one FP32 quotient and one correction
        // from the double-float residual b - g0 q (relative error ~2^-46)
        const DF b = df_mul_f(invc, pr.v);
        const DF q = df_add(DF{1.f, 0.f}, b);
        const float g0 = __fdiv_rn(b.hi, q.hi);
        const DF res = df_add(b, df_neg(df_mul_f(q, g0)));
        const DF g = df_norm(g0, __fdiv_rn(res.hi, q.hi));
        const DF A = df_add(Az, df_neg(df_mul(Az, g)));
        DF B = df_add(Bz, df_neg(df_mul(L, g)));
        if (P.resample) B = df_add(B, DF{-0.5f * A.hi, -0.5f * A.lo});
        const float t_last = fmaf(A.hi, t_lastj, B.hi);
        int bi = 0;
        float bf = 0.f, a_hi = 0.f, a_lo = 0.f;
        if (!(q.hi > 0.f) || !(B.hi < (float)n_ls) || !(t_last >= -1.f) || !(B.hi > -32768.f)) {
            // the spectrum misses every output bin (a_hi = 0 marks the record)
            r.w[0] = r.w[1] = r.w[2] = r.w[3] = 0.f;
        } else {
            // B = bi + bf, bf in [0, 1] rounded once; A = a_hi + a_lo with
            // a_hi of 11 significant bits, so that j a_hi is exact in FP32
            const float fb = floorf(B.hi);
            bi = (int)fb;
            bf = __fadd_rn(__fsub_rn(B.hi, fb), B.lo);
            if (bf < 0.f) {
                bf += 1.f;
                --bi;
            }
            a_hi = __uint_as_float(__float_as_uint(A.hi) & ~((1u << 13) - 1u));
            a_lo = __fadd_rn(__fsub_rn(A.hi, a_hi), A.lo);
        }
        mr.c0_bi = (c0 << 16) | (bi & 0xffff);
        mr.bf = bf;
        mr.a_hi = a_hi;
        mr.a_lo = a_lo;
        // Doppler shift in fixed point, and which rounds the particle takes
        const DF S = df_neg(df_mul(Ls, g)), D = df_neg(df_mul(Az, g));
        r.s0 = df_fixed(S, sc);
        r.g = df_fixed(D, scg);
        const float Af = a_hi + a_lo, delta = (1.f - a_hi) - a_lo;
        r.d = P.kind == 0 ? delta : D.hi;
        const float s_a = fmaf(-(float)P.jc, D.hi, S.hi), s_b = fmaf((float)(P.n_lambda - P.jc), D.hi, S.hi);
        const bool fits = Af > 0.f && Af <= P.a_max && fabsf(D.hi * scg) < 2147483000.f && fminf(s_a, s_b) >= P.s_min && fmaxf(s_a, s_b) <= P.s_max;
        const bool edges = Af >= 0.5f && Af < 1.999f;  // two-read edges (bin means)
        unsigned path = kPathBins;
        if (fits && P.kind == 0 && delta >= 0.f && delta * 31.f < 1.f) path = kPathMain;
        else if (fits && P.resample) path = !edges ? kPathBins : (P.kind == 0 ? kPathTwoRead : kPathMain);
        else if (fits) path = P.kind == 2 || (P.kind == 1 && Af >= 0.5f && delta > kShuffleTol) ? kPathMain : kPathTwoRead;
        const int e = path == kPathBins ? 0 : (ia - age_band(ia, P.apb, P.n_bands) * P.apb) * nzc + iz;
        r.ef = (unsigned)(8 * e) | (path << 30);
        P.map[i] = mr;
        P.rec[i] = r;
        if (P.prec) P.prec[i] = pr;
    }
}

int launch_setup(const SetupParams& P, long long n_total, cudaStream_t st) {
    if (n_total <= 0) return 0;
    long long nb = (n_total + 255) / 256;
    if (nb > 16ll * sm_count()) nb = 16ll * sm_count();
    k_setup<<<(int)nb, 256, 0, st>>>(P);
    return 1;
}

// ----------------------------------------------------------------------------
// Template layout (once per SSP grid): consecutive threads write consecutive
// entries of a node row and read n_age * n_Z rows of templates (25 MB written
// for the 50 x 10 x 3721 grid; on the host this took milliseconds).
// ----------------------------------------------------------------------------
__global__ void k_build_pairs(const SlabParams G, int apb, int n_age, int n_Z, const float* __restrict__ t,
                              void* __restrict__ pair, float2* __restrict__ adj) {
    const int nzc = max(n_Z, 2), ca = max(n_age - 1, 1);
    const long long total = G.band_stride * G.n_bands;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < total;
         i += (long long)gridDim.x * blockDim.x) {
        const int band = (int)(i / G.band_stride);
        const long long r = i - band * G.band_stride;
        const int k = (int)(r / G.pitch) - G.pad, e = (int)(r % G.pitch);
        const int ia = band * apb + e / nzc, iz = min(e % nzc, n_Z - 1);
        float v0 = 0.f, v1 = 0.f;  // zero rows outside the templates, zero entries past the band's
        if (k >= 0 && k < G.n_ls && e < apb * nzc && ia < ca) {
            v0 = t[((long long)ia * n_Z + iz) * G.n_ls + k];
            v1 = t[((long long)min(ia + 1, n_age - 1) * n_Z + iz) * G.n_ls + k];
        }
        if (G.qdt == 1) {
            const __nv_bfloat16 a = __float2bfloat16_rn(v0), b = __float2bfloat16_rn(v1);
            static_cast<uint32_t*>(pair)[i] = __bfloat16_as_ushort(a) | ((uint32_t)__bfloat16_as_ushort(b) << 16);
            v0 = __bfloat162float(a);
            v1 = __bfloat162float(b);
        } else if (G.qdt == 2) {
            const __half a = __float2half_rn(v0), b = __float2half_rn(v1);
            static_cast<uint32_t*>(pair)[i] = __half_as_ushort(a) | ((uint32_t)__half_as_ushort(b) << 16);
            v0 = __half2float(a);
            v1 = __half2float(b);
        } else {
            static_cast<float2*>(pair)[i] = make_float2(v0, v1);
        }
        if (adj) adj[i] = make_float2(v0, G.kind == 0 ? v1 : v1 - v0);
    }
}

int launch_build_pairs(const SlabParams& G, int apb, int n_age, int n_Z, const float* t, void* pair, float2* adj,
                       cudaStream_t st) {
    k_build_pairs<<<16 * sm_count(), 256, 0, st>>>(G, apb, n_age, n_Z, t, pair, adj);
    return 1;
}

// ----------------------------------------------------------------------------
// Work items: one per <= chunk particles of a spaxel (all age bands), in one
// launch over a chained scan (common.cuh) of the spaxels' items and partial
// rows. Empty spaxels get no item: k_rows writes their rows. (Counts, two scans
// of three launches and the fill were eight launches.)
// ----------------------------------------------------------------------------
constexpr int kItemTile = 1024;  // spaxels per block, one per thread

size_t item_chain_words(int n_s) { return chain_words(((long long)n_s + kItemTile) / kItemTile) + 1; }

__global__ void __launch_bounds__(kItemTile) k_items(const ItemParams P, int n_tiles) {
    __shared__ ChainShared sh;
    const unsigned tile = chain_ticket(P.chain, sh);
    if (tile == 0 && threadIdx.x == 0 && P.slow_count) *P.slow_count = 0ull;
    const int nb = P.n_bands;
    const long long s = (long long)tile * kItemTile + threadIdx.x;  // entry n_s closes the offsets
    int b0 = 0, e0 = 0;
    if (s < P.n_s) {
        b0 = P.seg_off[s * nb];
        e0 = P.seg_off[(s + 1) * nb];
    }
    const int ni = (e0 - b0 + P.chunk - 1) / P.chunk;
    const int np = ni > 1 ? ni : 0;  // partial rows
    // items below, partial rows from bit kPartShift (at most 2^24 + 2^24 of each:
    // spaxels, and particles / chunk)
    constexpr int kPartShift = 26, kLow = (1 << kPartShift) - 1;
    const unsigned long long pre =
        chain_exclusive(((unsigned long long)np << kPartShift) | (unsigned)ni, tile, P.chain, sh, kChainLong, P.quiet_scan);
    // a wait that ran out: offsets too small, so that items are lost, but every
    // offset stays within its buffers and readers check what the items hold
    if (pre >= kChainMissing) atomicOr(P.err, kErrTmaTimeout);
    if (s > P.n_s) return;
    const int base = (int)pre & kLow, part = (int)(pre >> kPartShift) & kLow;
    P.item_off[s] = base;
    P.part_off[s] = part;
    if (np) P.split[atomicAdd(P.chain + n_tiles + 1, 1ull)] = (int)s;
    for (int i = 0; i < ni; ++i) {
        if ((long long)base + i >= P.item_cap) {
            atomicOr(P.err, kErrBadItem);
            return;
        }
        Item it;
        it.spaxel = (int)s;
        it.begin = b0 + i * P.chunk;
        it.end = min(b0 + (i + 1) * P.chunk, e0);
        it.part_row = np ? part + i : -1;
        P.items[base + i] = it;
    }
}

int launch_items(const ItemParams& P, cudaStream_t st) {
    const int n_tiles = (int)(((long long)P.n_s + kItemTile) / kItemTile);  // covers entry n_s
    k_items<<<n_tiles, kItemTile, 0, st>>>(P, n_tiles);
    return 1;
}

}  // namespace rubix
