// engine.cu -- host side of the forward model: SSP state + deposit tiling,
// per-galaxy plans, and the enqueue sequence of one forward (see engine.h).
#include <algorithm>
#include <cmath>
#include <cstdarg>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <mutex>
#include <string>
#include <vector>

#include "engine.h"
#include "sort_layout.h"
#include "tile.cuh"

namespace rubix {

// ----------------------------------------------------------------------------
// errors
// ----------------------------------------------------------------------------
static thread_local std::string g_err;

rubix_status fail(rubix_status st, const char* fmt, ...) {
    char buf[512];
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(buf, sizeof(buf), fmt, ap);
    va_end(ap);
    g_err = buf;
    return st;
}
void set_last_error(const char* msg) { g_err = msg; }
const char* last_error() { return g_err.c_str(); }

#define CK(call)                                                                                          \
    do {                                                                                                  \
        cudaError_t e_ = (call);                                                                          \
        if (e_ != cudaSuccess)                                                                            \
            return fail(e_ == cudaErrorMemoryAllocation ? RUBIX_ERR_OOM : RUBIX_ERR_CUDA, "%s: %s (%s:%d)", \
                        #call, cudaGetErrorString(e_), __FILE__, __LINE__);                                \
    } while (0)

// ----------------------------------------------------------------------------
// helpers
// ----------------------------------------------------------------------------
namespace {

typedef CUresult (*PFN_encodeTiled_t)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                      const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                      CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

PFN_encodeTiled_t get_encode_tiled() {
    static PFN_encodeTiled_t fn = nullptr;
    static std::once_flag once;
    std::call_once(once, [] {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<PFN_encodeTiled_t>(p);
    });
    return fn;
}

void gauss_kernel(double sigma, int r, float* out) {
    std::vector<double> k(2 * r + 1);
    double s = 0.0;
    for (int d = -r; d <= r; ++d) {
        k[d + r] = std::exp(-(double)d * d / (2.0 * sigma * sigma));
        s += k[d + r];
    }
    for (int d = -r; d <= r; ++d) out[d + r] = (float)(k[d + r] / s);
}

int kernel_radius(double sigma, int r) {
    if (r > 0) return r;
    if (!(sigma > 0.0)) return 0;
    return (int)std::ceil(4.0 * sigma);
}

template <typename T>
cudaError_t dalloc_sync(T** p, size_t count) {
    *p = nullptr;
    if (count == 0) count = 1;
    return cudaMalloc(reinterpret_cast<void**>(p), count * sizeof(T));
}

}  // namespace

int sm_count() {
    static int cache[64] = {};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0) return 1;
    if (dev >= 64) {
        int n = 0;
        cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
        return n > 0 ? n : 1;
    }
    int n = __atomic_load_n(&cache[dev], __ATOMIC_RELAXED);
    if (n <= 0) {
        cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
        if (n <= 0) n = 1;
        __atomic_store_n(&cache[dev], n, __ATOMIC_RELAXED);
    }
    return n;
}

// ----------------------------------------------------------------------------
// validation
// ----------------------------------------------------------------------------
rubix_status validate_ssp(const rubix_ssp_grid* ssp) {
    if (!ssp) return fail(RUBIX_ERR_INVALID_ARG, "ssp is NULL");
    if (ssp->n_age < 1 || ssp->n_Z < 1 || ssp->n_lambda < 2 || ssp->n_lambda > 16384)
        return fail(RUBIX_ERR_INVALID_ARG, "SSP sizes out of range (n_age, n_Z >= 1, 2 <= n_lambda <= 16384)");
    if ((long long)ssp->n_age * ssp->n_Z > 65535) return fail(RUBIX_ERR_INVALID_ARG, "more than 65535 templates");
    if (!ssp->log10_age_nodes || !ssp->log10_Z_nodes || !ssp->spectra)
        return fail(RUBIX_ERR_INVALID_ARG, "SSP arrays must be non-NULL host pointers");
    for (int i = 1; i < ssp->n_age; ++i)
        if (!(ssp->log10_age_nodes[i] > ssp->log10_age_nodes[i - 1]))
            return fail(RUBIX_ERR_INVALID_ARG, "age nodes not strictly increasing");
    for (int i = 1; i < ssp->n_Z; ++i)
        if (!(ssp->log10_Z_nodes[i] > ssp->log10_Z_nodes[i - 1]))
            return fail(RUBIX_ERR_INVALID_ARG, "Z nodes not strictly increasing");
    if (!(ssp->dlambda > 0.0)) return fail(RUBIX_ERR_INVALID_ARG, "SSP dlambda must be > 0");
    if (ssp->storage_dtype < 0 || ssp->storage_dtype > 2) return fail(RUBIX_ERR_INVALID_ARG, "bad storage_dtype");
    return RUBIX_OK;
}

rubix_status validate_telescope(const rubix_telescope* tel, double ssp_dlambda) {
    if (!tel) return fail(RUBIX_ERR_INVALID_ARG, "telescope is NULL");
    if (tel->nx < 1 || tel->ny < 1 || tel->ny > 65535 || (long long)tel->nx * tel->ny >= (1ll << 24))
        return fail(RUBIX_ERR_INVALID_ARG, "nx, ny out of range (ny <= 65535, nx*ny < 2^24)");
    if (!(tel->spaxel_size > 0.0)) return fail(RUBIX_ERR_INVALID_ARG, "spaxel_size must be > 0");
    if (tel->n_lambda < 1 || tel->n_lambda > 8192) return fail(RUBIX_ERR_INVALID_ARG, "n_lambda must be in [1, 8192]");
    if (!(tel->dlambda > 0.0)) return fail(RUBIX_ERR_INVALID_ARG, "dlambda must be > 0");
    if (!(tel->psf_fwhm >= 0.0) || !(tel->lsf_sigma >= 0.0)) return fail(RUBIX_ERR_INVALID_ARG, "negative PSF/LSF width");
    if (!(tel->z_cosmo > -1.0)) return fail(RUBIX_ERR_INVALID_ARG, "z_cosmo must be > -1");
    if (tel->resample != 0 && tel->resample != 1) return fail(RUBIX_ERR_INVALID_ARG, "resample must be 0 or 1");
    if (!(tel->row_lo == 0 && tel->row_hi == 0) && !(tel->row_lo >= 0 && tel->row_lo < tel->row_hi && tel->row_hi <= tel->ny))
        return fail(RUBIX_ERR_INVALID_ARG, "row window must satisfy 0 <= row_lo < row_hi <= ny (or 0, 0 for all rows)");
    if (tel->dlambda / ((1.0 + tel->z_cosmo) * ssp_dlambda) > 3.0)
        return fail(RUBIX_ERR_INVALID_ARG, "instrument bins wider than 3 SSP steps are not supported");
    const double sp = tel->psf_fwhm / (2.0 * std::sqrt(2.0 * std::log(2.0)));
    const double sl = tel->lsf_sigma / tel->dlambda;
    if ((sp > 0.0 && kernel_radius(sp, tel->psf_radius) > kMaxRadius) ||
        (sl > 0.0 && kernel_radius(sl, tel->lsf_radius) > kMaxRadius))
        return fail(RUBIX_ERR_INVALID_ARG, "PSF/LSF radius > 64");
    return RUBIX_OK;
}

rubix_status check_particles(const rubix_particles* p) {
    if (!p) return fail(RUBIX_ERR_INVALID_ARG, "particles is NULL");
    if (p->n < 0 || p->n > (1ll << 30)) return fail(RUBIX_ERR_INVALID_ARG, "n out of range");
    if (p->n == 0) return RUBIX_OK;
    if (!p->x || !p->y || !p->mass || !p->age || !p->Z) return fail(RUBIX_ERR_INVALID_ARG, "x, y, mass, age, Z required");
    if (p->preprojected) {
        if (!p->v_los) return fail(RUBIX_ERR_INVALID_ARG, "v_los required when preprojected");
    } else {
        if (!p->z || !p->vy || !p->vz) return fail(RUBIX_ERR_INVALID_ARG, "z, vy, vz required when not preprojected");
        if (!p->vx && p->azimuth != 0.0) return fail(RUBIX_ERR_INVALID_ARG, "vx required when azimuth != 0");
    }
    return RUBIX_OK;
}

void orientation_matrix(double inclination, double azimuth, double position_angle, double R[9], double Di[3],
                        double Da[2]) {
    const double ca = std::cos(azimuth), sa = std::sin(azimuth);
    const double ci = std::cos(inclination), si = std::sin(inclination);
    const double cq = std::cos(position_angle), sq = std::sin(position_angle);
    const double cisa = ci * sa, cica = ci * ca;
    R[0] = cq * ca - sq * cisa;
    R[1] = -(cq * sa) - sq * cica;
    R[2] = sq * si;
    R[3] = sq * ca + cq * cisa;
    R[4] = cq * cica - sq * sa;
    R[5] = -(cq * si);
    R[6] = si * sa;
    R[7] = si * ca;
    R[8] = ci;
    Di[0] = cisa;
    Di[1] = cica;
    Di[2] = -si;
    Da[0] = si * ca;
    Da[1] = -(si * sa);
}

int window_rows(const rubix_telescope* tel) { return (tel->row_hi > 0) ? tel->row_hi - tel->row_lo : tel->ny; }

bool same_wavelength_grid(const SspState& S, const rubix_telescope* tel) {
    return tel->n_lambda == S.n_lambda && tel->lambda0 == S.lambda0 && tel->dlambda == S.dlambda &&
           tel->z_cosmo == S.z_cosmo;
}

// ----------------------------------------------------------------------------
// SSP state
// ----------------------------------------------------------------------------
void ssp_state_destroy(SspState* S) {
    if (!S) return;
    int prev = 0;
    cudaGetDevice(&prev);
    cudaSetDevice(S->device);
    void* ptrs[] = {S->d_pair, S->d_pair_adj, S->d_la, S->d_lz, S->d_tile_klo, S->d_tile_ref, S->d_lane_ref, S->d_err, S->d_slow};
    for (void* p : ptrs)
        if (p) cudaFree(p);
    cudaSetDevice(prev);
    delete S;
}

rubix_status ssp_state_create(const rubix_ssp_grid* ssp, const rubix_telescope* tel, bool with_adjoint,
                              SspState** out) {
    *out = nullptr;
    rubix_status st = validate_ssp(ssp);
    if (st != RUBIX_OK) return st;
    st = validate_telescope(tel, ssp->dlambda);
    if (st != RUBIX_OK) return st;
    SspState* h = new SspState();
    auto bail = [&](rubix_status s) {
        ssp_state_destroy(h);
        return s;
    };
    if (cudaGetDevice(&h->device) != cudaSuccess) return bail(fail(RUBIX_ERR_CUDA, "no CUDA device"));
    cudaDeviceGetAttribute(&h->n_sm, cudaDevAttrMultiProcessorCount, h->device);
    cudaDeviceGetAttribute(&h->smem_optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, h->device);
    h->n_lambda = tel->n_lambda;
    h->lambda0 = tel->lambda0;
    h->dlambda = tel->dlambda;
    h->z_cosmo = tel->z_cosmo;

    // ---- SSP grid: sizes and node vectors (the templates go to the device as
    // age pairs, below) ----
    SspDev& S = h->ssp;
    S.dtype = ssp->storage_dtype;
    S.n_age = ssp->n_age;
    S.n_Z = ssp->n_Z;
    S.n_t = ssp->n_age * ssp->n_Z;
    S.n_ls = ssp->n_lambda;
    S.ls0 = ssp->lambda0;
    S.dls = ssp->dlambda;
    {
        std::vector<float> la(S.n_age), lz(S.n_Z);
        for (int i = 0; i < S.n_age; ++i) la[i] = (float)ssp->log10_age_nodes[i];
        for (int i = 0; i < S.n_Z; ++i) lz[i] = (float)ssp->log10_Z_nodes[i];
        if (dalloc_sync(&h->d_la, S.n_age) || dalloc_sync(&h->d_lz, S.n_Z) || dalloc_sync(&h->d_err, 4) ||
            dalloc_sync(&h->d_slow, 1))
            return bail(fail(RUBIX_ERR_OOM, "SSP state alloc"));
        cudaMemcpy(h->d_la, la.data(), la.size() * 4, cudaMemcpyHostToDevice);
        cudaMemcpy(h->d_lz, lz.data(), lz.size() * 4, cudaMemcpyHostToDevice);
        cudaMemset(h->d_err, 0, 16);
        cudaMemset(h->d_slow, 0, 8);
        S.la_nodes = h->d_la;
        S.lz_nodes = h->d_lz;
    }

    // ---- deposit tiling: wavelength tiles and the slab staged per tile and age band ----
    const SlabLayout L = slab_layout(S.n_age, S.n_Z, S.ls0, S.dls, tel->n_lambda, tel->lambda0, tel->dlambda, tel->z_cosmo,
                                     ((long long)h->smem_optin - kDepHeader) / (long long)sizeof(float2),
                                     RUBIX_DEP_VHALO / kC_kms, RUBIX_DEP_BANDS);
    const int ca = std::max(S.n_age - 1, 1);
    h->apb = L.apb;
    SlabParams& G = h->geo;
    G.kind = L.kind;
    G.n_bands = L.n_bands;
    G.pitch = L.pitch;
    G.slab_w = L.slab_w;
    G.need = L.need;
    G.a_max = L.a_max;
    G.tile_w = L.tile_w;
    G.n_tiles = L.n_tiles;
    G.n_lambda = tel->n_lambda;
    G.n_ls = S.n_ls;
    G.es = S.n_Z > 1 ? 1 : 2;
    G.pad = G.slab_w + 8;
    for (int m = 0; m < 2; ++m) {
        G.ib[m] = L.ib[m];
        G.fbr[m] = L.fbr[m];
    }
    G.a0_1m = L.a0_1m;
    G.fb = L.fb;
    G.jc = L.jc;
    G.s_min = L.s_min;
    G.s_max = L.s_max;
    G.cost_c0 = RUBIX_DEP_COSTC0;
    for (int b = 0; b < kMaxBands; ++b) G.band_e0[b] = std::min(b * L.apb, ca - 1) * L.nzc;
    std::vector<float2> lref;
    for (int l = 0; l < 32; ++l) lref.push_back(make_float2(L.lane_node[l], L.lane_rest[l]));
    if (dalloc_sync(&h->d_tile_klo, G.n_tiles) || dalloc_sync(&h->d_tile_ref, 2 * (size_t)G.n_tiles) ||
        dalloc_sync(&h->d_lane_ref, 32))
        return bail(fail(RUBIX_ERR_OOM, "tile alloc"));
    cudaMemcpy(h->d_tile_klo, L.klo.data(), L.klo.size() * 4, cudaMemcpyHostToDevice);
    cudaMemcpy(h->d_tile_ref, L.tile_ref.data(), L.tile_ref.size() * 4, cudaMemcpyHostToDevice);
    cudaMemcpy(h->d_lane_ref, lref.data(), 32 * sizeof(float2), cudaMemcpyHostToDevice);
    G.tile_ref = h->d_tile_ref;
    G.lane_ref = h->d_lane_ref;
    G.tile_klo = h->d_tile_klo;
    h->dep_smem = deposit_smem_bytes(G.pitch, G.slab_w);
    h->dep_ctas = h->n_sm;
    G.err = h->d_err;

    // ---- age pairs: entry (ia, iz) of node k holds templates (ia, iz) and
    // (ia + 1, iz), so that a cell's four corners are entries iz and iz + 1 (a
    // grid of one metallicity repeats its entry). One block per age band,
    // node-major, pad zero node rows on both sides, in the storage dtype: FP32
    // pairs, or two BF16 / FP16 bit patterns (first | second << 16) that the
    // kernels widen to FP32 exactly; laid out on the device (k_build_pairs) ----
    G.qdt = (S.dtype == RUBIX_F32) ? 0 : (S.dtype == RUBIX_BF16 ? 1 : 2);
    static_assert(kDepHeader % 128 == 0, "slab must start 16-byte aligned");
    {
        const size_t rows = (size_t)S.n_ls + 2 * (size_t)G.pad;
        G.band_stride = (long long)((rows * G.pitch + 3) / 4 * 4);
        const size_t total = (size_t)G.band_stride * G.n_bands, nt = (size_t)S.n_age * S.n_Z * S.n_ls;
        std::vector<float> tf(nt);
        for (size_t i = 0; i < nt; ++i) tf[i] = (float)ssp->spectra[i];
        const bool own_adj = with_adjoint && !(G.kind == 0 && G.qdt == 0);  // else d_pair serves
        float* d_t = nullptr;
        const bool ok = cudaMalloc(&h->d_pair, total * (G.qdt ? 4 : 8)) == cudaSuccess &&
                        (!own_adj || dalloc_sync(&h->d_pair_adj, total) == cudaSuccess) &&
                        dalloc_sync(&d_t, nt) == cudaSuccess;
        cudaError_t e = cudaSuccess;
        if (ok) {
            G.pair = h->d_pair;
            e = cudaMemcpy(d_t, tf.data(), nt * sizeof(float), cudaMemcpyHostToDevice);
            if (e == cudaSuccess) {
                launch_build_pairs(G, L.apb, S.n_age, S.n_Z, d_t, h->d_pair, h->d_pair_adj, nullptr);
                e = cudaDeviceSynchronize();
            }
        }
        if (d_t) cudaFree(d_t);
        cudaGetLastError();
        if (!ok) return bail(fail(RUBIX_ERR_OOM, "template alloc"));
        if (e != cudaSuccess) return bail(fail(RUBIX_ERR_CUDA, "template copy: %s", cudaGetErrorString(e)));
    }
    if (cudaDeviceSynchronize() != cudaSuccess)
        return bail(fail(RUBIX_ERR_CUDA, "SSP state: %s", cudaGetErrorString(cudaGetLastError())));
    *out = h;
    return RUBIX_OK;
}

// ----------------------------------------------------------------------------
// plans
// ----------------------------------------------------------------------------
namespace {

struct Buf {
    void** ptr;
    size_t bytes;
};

// Particles per work item of a galaxy of n: RUBIX_DEP_CHUNK, or less where that
// would leave a warp of the deposit fewer than about eight full items a forward,
// too few to even out their lengths (5e5 particles on the survey grid: 976 us
// with 256, 872 with 64; 2e5 particles, gradient step with bin means: 3.72 and
// 3.60 ms; on the mid-size and large galaxies smaller items cost 1 - 5 %). It
// depends on the request alone, so that its cube does not depend on the plan.
int item_chunk(const SspState& S, long long n, bool compact) {
    if (compact) return RUBIX_DEP_CHUNK;
    const double items = (double)n * S.geo.n_tiles / ((double)S.n_sm * (S.dep_threads / 32) * 8.0);
    int c = RUBIX_DEP_CHUNK;
    while (c > RUBIX_DEP_CHUNK / 4 && c > items) c /= 2;
    return c;
}
// The most of n' / item_chunk(n') over n' <= n (the smaller chunks end at a
// known count).
long long max_chunks(const SspState& S, long long n, bool compact) {
    if (compact) return n / RUBIX_DEP_CHUNK;
    const long long lim = (long long)RUBIX_DEP_CHUNK * S.n_sm * (S.dep_threads / 32) * 8 / std::max(S.geo.n_tiles, 1) + 1;
    return std::max(n / RUBIX_DEP_CHUNK, std::min(n, lim) / (RUBIX_DEP_CHUNK / 4));
}
// Partial rows: ceil(count / chunk) of each split spaxel, each of more than chunk
// particles.
long long max_parts(const SspState& S, int n_s, long long n, bool compact) {
    const long long c = max_chunks(S, n, compact);
    return c + std::min<long long>(n_s, c) + 2;
}

// Every device buffer of a plan for n particles, with its size.
std::vector<Buf> plan_buffers(Plan* P, const SspState& S, int n_s, int n_lambda, long long n, bool with_out,
                              bool with_grad, bool need_tmp, bool staging, int pitch0, bool compact) {
    const size_t N = (size_t)std::max(n, 1ll);
    const long long item_cap = (long long)n_s + max_chunks(S, n, compact) + 2;
    const long long part_cap = max_parts(S, n_s, n, compact);
    const size_t cube = (size_t)n_s * n_lambda * sizeof(float);
    std::vector<Buf> v;
    if (staging)
        v = {{(void**)&P->d_x, 4 * N},    {(void**)&P->d_y, 4 * N},    {(void**)&P->d_z, 4 * N},
             {(void**)&P->d_vx, 4 * N},   {(void**)&P->d_vy, 4 * N},   {(void**)&P->d_vz, 4 * N},
             {(void**)&P->d_vlos, 4 * N},
             {(void**)&P->d_mass, 4 * N}, {(void**)&P->d_age, 4 * N}, {(void**)&P->d_Z, 4 * N}};
    const std::vector<Buf> rest = {
        {(void**)&P->d_key, 4 * N},
        {(void**)&P->d_keys_tmp, 4 * N}, {(void**)&P->d_vals_tmp, 4 * N}, {(void**)&P->d_skeys, 4 * N},
        {(void**)&P->d_perm, 4 * N}, {(void**)&P->d_pin, 16 * N},
        {(void**)&P->d_sort_scratch, 4 * sort_scratch_ints((long long)N, S.n_sm, compact)},
        {(void**)&P->d_items, sizeof(Item) * (size_t)item_cap}, {(void**)&P->d_rec, sizeof(DepRec) * N},
        {(void**)&P->d_map, sizeof(MapRec) * N},
        {(void**)&P->d_partials, 4 * (size_t)part_cap * n_lambda},
        {(void**)&P->d_seg_off, 4 * ((size_t)n_s * S.geo.n_bands + 2)},
        {(void**)&P->d_item_off, 4 * ((size_t)n_s + 1)}, {(void**)&P->d_part_off, 4 * ((size_t)n_s + 1)},
        {(void**)&P->d_split, 4 * (size_t)n_s}, {(void**)&P->d_chain, 8 * item_chain_words(n_s)},
        {(void**)&P->d_cube0, (size_t)n_s * std::max(pitch0, n_lambda) * sizeof(float)},
    };
    v.insert(v.end(), rest.begin(), rest.end());
    if (need_tmp) v.push_back({(void**)&P->d_tmp, cube});
    if (with_out) v.push_back({(void**)&P->d_out, cube});
    if (with_grad) {
        v.push_back({(void**)&P->d_prec, sizeof(PartRec) * N});
        v.push_back({(void**)&P->d_contrib, 8 * kGlobal * N});
        v.push_back({(void**)&P->d_dvda, 8 * N});
        v.push_back({(void**)&P->d_red, 8 * 1024});
        v.push_back({(void**)&P->d_wu, 8 * N});
        v.push_back({(void**)&P->d_adjpart, 16 * N * (size_t)std::max(S.geo.n_tiles, 1)});
    }
    return v;
}

size_t round256(size_t b) { return (b + 255) / 256 * 256; }

int conv_radius_psf(const rubix_telescope* tel) {
    const double sp = tel->psf_fwhm / (2.0 * std::sqrt(2.0 * std::log(2.0)));
    return sp > 0.0 ? kernel_radius(sp, tel->psf_radius) : 0;
}
// Row stride of the pre-convolution cube: 16-byte rows when the PSF/LSF radii
// have a TMA kernel (it loads rows with 3-D TMA boxes), else dense.
int cube0_pitch(int rp, int rl, int n_lambda) {
    unsigned box[2];
    return conv_tma_box(rp, rl, box) ? (n_lambda + 3) / 4 * 4 : n_lambda;
}

int conv_radius_lsf(const rubix_telescope* tel) {
    const double sl = tel->lsf_sigma / tel->dlambda;
    return sl > 0.0 ? kernel_radius(sl, tel->lsf_radius) : 0;
}

}  // namespace

bool conv_params(const rubix_telescope* tel, int rows, ConvParams* C) {
    C->nx = tel->nx;
    C->ny = rows;
    C->n_lambda = tel->n_lambda;
    const double sp = tel->psf_fwhm / (2.0 * std::sqrt(2.0 * std::log(2.0)));
    const double sl = tel->lsf_sigma / tel->dlambda;
    C->rp = conv_radius_psf(tel);
    C->rl = conv_radius_lsf(tel);
    if (sp > 0.0) gauss_kernel(sp, C->rp, C->gp); else C->gp[0] = 1.f;
    if (sl > 0.0) gauss_kernel(sl, C->rl, C->gl); else C->gl[0] = 1.f;
    C->noise_inv_s2n = 0.f;
    return (sp > 0.0) || (sl > 0.0);
}

size_t plan_bytes(const SspState& S, const rubix_telescope* tel, long long n, bool with_out, bool with_grad,
                  bool staging, bool compact) {
    Plan tmp;
    const int rp = conv_radius_psf(tel), rl = conv_radius_lsf(tel);
    const bool need_tmp = psf_lsf_needs_tmp(rp, rl);
    size_t total = 0;
    for (const Buf& b : plan_buffers(&tmp, S, tel->nx * window_rows(tel), tel->n_lambda, n, with_out, with_grad, need_tmp,
                                     staging, cube0_pitch(rp, rl, tel->n_lambda), compact))
        total += round256(b.bytes);
    return total;
}

void plan_release(Plan* P) {
    if (!P->S) return;
    const bool need_tmp = true;
    for (const Buf& b : plan_buffers(P, *P->S, P->n_s, P->tel.n_lambda, P->cap, true, true, need_tmp, true, P->pitch0,
                                     P->alloc.compact)) {
        if (*b.ptr) {
            if (P->alloc.async) cudaFreeAsync(*b.ptr, P->alloc.stream);
            else cudaFree(*b.ptr);
        }
        *b.ptr = nullptr;
    }
    P->bytes = 0;
    P->cap = 0;
}

// Host-side fault injection for tests: RUBIX_FAULT_ALLOC_AT=k makes the k-th
// buffer allocation of every plan fail as if the device were out of memory
// (nothing is run on the GPU; the plan's other buffers are released).
static int fault_alloc_at() {
    const char* e = std::getenv("RUBIX_FAULT_ALLOC_AT");
    return e ? std::atoi(e) : 0;
}

// RUBIX_FAULT_SCAN (tests): the blocks of a plan's scans publish nothing, so that
// every wait in them runs out: 1 the sort's, 2 the work items'.
static int fault_scan() {
    const char* e = std::getenv("RUBIX_FAULT_SCAN");
    return e ? std::atoi(e) : 0;
}

rubix_status plan_init(Plan* P, const SspState* S, const rubix_telescope* tel, long long n, Alloc a, bool with_out,
                       bool with_grad) {
    rubix_status st = validate_telescope(tel, S->ssp.dls);
    if (st != RUBIX_OK) return st;
    if (!same_wavelength_grid(*S, tel))
        return fail(RUBIX_ERR_INVALID_ARG, "telescope wavelength grid differs from the SSP state's");
    if (n < 0 || n > (1ll << 30)) return fail(RUBIX_ERR_INVALID_ARG, "particle count out of range");
    P->S = S;
    P->quiet_scan = fault_scan();
    P->alloc = a;
    P->tel = *tel;
    if (P->tel.flux_scale == 0.0) P->tel.flux_scale = 1.0;
    P->rows = window_rows(tel);
    P->row_lo = (tel->row_hi > 0) ? tel->row_lo : 0;
    P->n_s = tel->nx * P->rows;
    P->x_lo = (-0.5 * (double)tel->nx) * tel->spaxel_size;
    P->y_lo = (-0.5 * (double)tel->ny) * tel->spaxel_size;
    P->inv_size = 1.0 / tel->spaxel_size;
    ConvParams& C = P->conv;
    P->need_conv = conv_params(tel, P->rows, &C);
    C.err = S->d_err;
    P->pitch0 = cube0_pitch(C.rp, C.rl, tel->n_lambda);
    P->has_conv_map = false;
    P->cap = std::max(n, 1ll);
    P->item_cap = (long long)P->n_s + max_chunks(*S, P->cap, a.compact) + 2;
    P->part_cap = max_parts(*S, P->n_s, P->cap, a.compact);
    const bool need_tmp = psf_lsf_needs_tmp(C.rp, C.rl);
    P->bytes = 0;
    const int fail_at = fault_alloc_at();
    int idx = 0;
    for (const Buf& b :
         plan_buffers(P, *S, P->n_s, tel->n_lambda, P->cap, with_out, with_grad, need_tmp, a.staging, P->pitch0,
                      a.compact)) {
        cudaError_t e;
        if (++idx == fail_at) e = cudaErrorMemoryAllocation;
        else if (!a.async) e = cudaMalloc(b.ptr, round256(b.bytes));
        else if (a.pool) e = cudaMallocFromPoolAsync(b.ptr, round256(b.bytes), a.pool, a.stream);
        else e = cudaMallocAsync(b.ptr, round256(b.bytes), a.stream);
        if (e != cudaSuccess) {
            *b.ptr = nullptr;
            cudaGetLastError();
            plan_release(P);
            return fail(RUBIX_ERR_OOM, "plan allocation of %zu bytes failed: %s", b.bytes, cudaGetErrorString(e));
        }
        P->bytes += round256(b.bytes);
    }
    unsigned box[2];
    if (P->need_conv && conv_tma_box(C.rp, C.rl, box)) {
        // 3-D view of the pre-convolution cube: x = bin (n_lambda of each
        // pitched row), y = spaxel x, z = spaxel y; zero fill outside
        PFN_encodeTiled_t enc = get_encode_tiled();
        if (!enc) {
            plan_release(P);
            return fail(RUBIX_ERR_CUDA, "cuTensorMapEncodeTiled unavailable");
        }
        cuuint64_t gdim[3] = {(cuuint64_t)tel->n_lambda, (cuuint64_t)tel->nx, (cuuint64_t)P->rows};
        cuuint64_t gstr[2] = {(cuuint64_t)P->pitch0 * 4, (cuuint64_t)P->pitch0 * 4 * (cuuint64_t)tel->nx};
        cuuint32_t bx[3] = {box[0], box[1], 1};
        cuuint32_t es[3] = {1, 1, 1};
        CUresult r = enc(&P->conv_map, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 3, P->d_cube0, gdim, gstr, bx, es,
                         CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                         CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
        if (r != CUDA_SUCCESS) {
            plan_release(P);
            return fail(RUBIX_ERR_CUDA, "cuTensorMapEncodeTiled (PSF/LSF) failed (%d)", (int)r);
        }
        P->has_conv_map = true;
    }
    return RUBIX_OK;
}

rubix_status plan_grow(Plan* P, long long n) {
    if (P->alloc.async) return fail(RUBIX_ERR_INVALID_ARG, "stream-ordered plans do not grow");
    const bool with_out = P->d_out != nullptr, with_grad = P->d_contrib != nullptr;
    const SspState* S = P->S;
    const rubix_telescope tel = P->tel;
    CK(cudaDeviceSynchronize());
    plan_release(P);
    return plan_init(P, S, &tel, n + n / 8, P->alloc, with_out, with_grad);
}

// ----------------------------------------------------------------------------
// forward, in enqueued parts
// ----------------------------------------------------------------------------
namespace {

// Host inputs are copied into the plan's staging buffers; device inputs are
// read in place. arrs[] follows rubix_particles' field order.
rubix_status stage_particles(Plan& P, const rubix_particles* p, const float** arrs, cudaStream_t st) {
    const long long n = p->n;
    const float* src[10] = {p->x, p->y, p->z, p->vx, p->vy, p->vz, p->v_los, p->mass, p->age, p->Z};
    float* dst[10] = {P.d_x, P.d_y, P.d_z, P.d_vx, P.d_vy, P.d_vz, P.d_vlos, P.d_mass, P.d_age, P.d_Z};
    for (int i = 0; i < 10; ++i) {
        arrs[i] = nullptr;
        if (!src[i] || n == 0) continue;
        if (p->on_device) {
            arrs[i] = src[i];
        } else if (!p->preprojected || i < 2 || i > 5) {
            // host arrays the call reads (the 3-D ones only for 3-D input)
            if (!dst[i]) return fail(RUBIX_ERR_INVALID_ARG, "host particle arrays need a plan with staging buffers");
            CK(cudaMemcpyAsync(dst[i], src[i], (size_t)n * 4, cudaMemcpyHostToDevice, st));
            arrs[i] = dst[i];
        }
    }
    if (p->preprojected) arrs[2] = arrs[3] = arrs[4] = arrs[5] = nullptr;
    else arrs[6] = nullptr;
    return RUBIX_OK;
}

AssignParams assign_params(const Plan& P, const rubix_particles* p, const float* const* arrs) {
    AssignParams A{};
    A.n = p->n;
    A.x = arrs[0];
    A.y = arrs[1];
    A.z = arrs[2];
    A.vx = arrs[3];
    A.vy = arrs[4];
    A.vz = arrs[5];
    A.v_los = arrs[6];
    A.preprojected = p->preprojected ? 1 : 0;
    orientation_matrix(p->inclination, p->azimuth, p->position_angle, A.R, A.Di, A.Da);
    A.x_lo = P.x_lo;
    A.y_lo = P.y_lo;
    A.inv_size = P.inv_size;
    A.nx = P.tel.nx;
    A.ny = P.tel.ny;
    A.row_lo = P.row_lo;
    A.rows = P.rows;
    A.n_bands = 1;
    return A;
}

}  // namespace

rubix_status enqueue_keys(Plan& P, const rubix_particles* p, int* keys_out, cudaStream_t st) {
    if (p->n > P.cap) return fail(RUBIX_ERR_INVALID_ARG, "more particles than the plan holds");
    if (p->n == 0) return RUBIX_OK;
    const float* arrs[10];
    rubix_status s = stage_particles(P, p, arrs, st);
    if (s != RUBIX_OK) return s;
    AssignParams A = assign_params(P, p, arrs);
    A.key = keys_out;
    A.pin_out = nullptr;
    launch_assign(A, st);
    CK(cudaGetLastError());
    return RUBIX_OK;
}

rubix_status enqueue_pre(Plan& P, const rubix_particles* p, cudaStream_t st, cudaEvent_t* ev) {
    NvtxRange nvtx("rubix: assign, sort, setup, items");
    const SspState& S = *P.S;
    if (p->n > P.cap) return fail(RUBIX_ERR_INVALID_ARG, "more particles than the plan holds");
    const long long n = p->n;
    const float* arrs[10];
    rubix_status s = stage_particles(P, p, arrs, st);
    if (s != RUBIX_OK) return s;
    P.launches = 0;
    P.dep_launches = 0;
    if (n > 0) {
        AssignParams A = assign_params(P, p, arrs);
        A.key = P.d_key;
        A.pin_out = P.d_pin;
        A.mass = arrs[7];
        A.Zm = arrs[9];
        A.dv_dang = P.d_dvda;  // null unless the plan keeps backward state
        A.age = arrs[8];
        A.la_nodes = S.d_la;
        A.n_age = S.ssp.n_age;
        A.apb = S.apb;
        A.n_bands = S.geo.n_bands;
        P.launches += launch_assign(A, st);
        const int ls = launch_sort_by_key(P.d_key, n, P.n_s * S.geo.n_bands + 1, P.d_keys_tmp, P.d_vals_tmp, P.d_skeys,
                                          P.d_perm, P.d_seg_off, P.d_sort_scratch, sort_scratch_ints(P.cap, S.n_sm, P.alloc.compact),
                                          P.alloc.compact, P.d_chain, (int)item_chain_words(P.n_s), P.quiet_scan == 1, st);
        if (ls < 0) return fail(RUBIX_ERR_CUDA, "internal: sort scratch too small for %lld particles", n);
        P.launches += ls;
    } else {
        CK(cudaMemsetAsync(P.d_chain, 0, 8 * item_chain_words(P.n_s), st));
        CK(cudaMemsetAsync(P.d_seg_off, 0, ((size_t)P.n_s * S.geo.n_bands + 2) * sizeof(int), st));
    }
    if (ev) cudaEventRecord(ev[1], st);
    SetupParams SP{};
    SP.ssp = S.ssp;
    SP.perm = P.d_perm;
    SP.seg_off = P.d_seg_off;
    SP.n_s = P.n_s;
    SP.n_bands = S.geo.n_bands;
    SP.pin = P.d_pin;
    SP.l0 = P.tel.lambda0;
    SP.dl = P.tel.dlambda;
    SP.z_cosmo = P.tel.z_cosmo;
    SP.inv_c = 1.0 / kC_kms;
    SP.alpha_z = 1.0 / ((1.0 + P.tel.z_cosmo) * S.ssp.dls);
    SP.ls0_dls = S.ssp.ls0 / S.ssp.dls;
    SP.flux_scale = P.tel.flux_scale;
    SP.n_lambda = P.tel.n_lambda;
    SP.resample = P.tel.resample;
    SP.rec = P.d_rec;
    SP.map = P.d_map;
    SP.fb = S.geo.fb;
    SP.jc = S.geo.jc;
    SP.apb = S.apb;
    SP.kind = S.geo.kind;
    SP.a_max = S.geo.a_max;
    SP.s_min = S.geo.s_min;
    SP.s_max = S.geo.s_max;
    SP.prec = P.d_prec;
    SP.n_cap = P.cap;
    P.launches += launch_setup(SP, n, st);
    ItemParams IP{};
    IP.seg_off = P.d_seg_off;
    IP.n_s = P.n_s;
    IP.n_bands = S.geo.n_bands;
    IP.chunk = item_chunk(S, n, P.alloc.compact);
    IP.item_off = P.d_item_off;
    IP.part_off = P.d_part_off;
    IP.items = P.d_items;
    IP.item_cap = P.item_cap;
    IP.split = P.d_split;
    IP.chain = P.d_chain;
    IP.quiet_scan = P.quiet_scan == 2;
    IP.slow_count = P.alloc.async ? nullptr : S.d_slow;  // one forward at a time on a handle
    IP.err = S.d_err;
    P.launches += launch_items(IP, st);
    P.last_n = n;
    CK(cudaGetLastError());
    return RUBIX_OK;
}

float* deposit_target(const Plan& P, float* out, bool noise) { return (P.need_conv || noise) ? P.d_cube0 : out; }

DepJob plan_job(const Plan& P, float* target) {
    DepJob J{};
    J.rec = P.d_rec;
    J.map = P.d_map;
    J.items = P.d_items;
    J.item_off = P.d_item_off;
    J.seg_off = P.d_seg_off;
    J.cube = target;
    J.partials = P.d_partials;
    J.part_cap = P.part_cap;
    J.n_s = P.n_s;
    J.pitch = (target == P.d_cube0) ? P.pitch0 : P.tel.n_lambda;
    J.resample = P.tel.resample;
    return J;
}

int enqueue_deposit(const SspState& S, const DepJob* jobs, int n_jobs, cudaStream_t st) {
    NvtxRange nvtx("rubix: deposit");
    if (n_jobs < 1 || n_jobs > kMaxJobs) return -1;
    DepositParams DP{};
    static_cast<SlabParams&>(DP) = S.geo;
    for (int j = 0; j < n_jobs; ++j) DP.jobs[j] = jobs[j];
    DP.n_jobs = n_jobs;
    DP.slow_count = S.d_slow;
    return launch_deposit(DP, S.dep_ctas, S.dep_threads, S.dep_smem, st);
}

int enqueue_post(Plan& P, float* target, float* out, uint64_t noise_seed, float noise_s2n, cudaStream_t st,
                 cudaEvent_t* ev) {
    NvtxRange nvtx("rubix: rows, PSF/LSF, noise");
    const int pitch = target == P.d_cube0 ? P.pitch0 : P.tel.n_lambda;
    const bool noise = noise_s2n > 0.f;
    // the fused convolution does not read rows out of every particle's reach
    const bool skip = target == P.d_cube0 && P.has_conv_map;
    RowParams RP{};
    RP.seg_off = P.d_seg_off;
    RP.nx = P.tel.nx;
    RP.ny = P.rows;
    RP.n_bands = P.S->geo.n_bands;
    RP.n_lambda = P.tel.n_lambda;
    RP.pitch = pitch;
    RP.skip_rp = skip ? P.conv.rp : -1;
    RP.part_off = P.d_part_off;
    RP.split = P.d_split;
    RP.n_split = P.d_chain + item_chain_words(P.n_s) - 1;
    RP.max_split = P.last_n / item_chunk(*P.S, P.last_n, P.alloc.compact);
    RP.partials = P.d_partials;
    RP.cube = target;
    int l = launch_rows(RP, st);
    if (ev) cudaEventRecord(ev[4], st);
    if (P.need_conv || noise) {
        ConvParams C = P.conv;
        C.seg_off = skip ? P.d_seg_off : nullptr;
        C.seg_bands = P.S->geo.n_bands;
        C.noise_inv_s2n = noise ? 1.0f / noise_s2n : 0.f;
        C.seed_lo = (uint32_t)noise_seed;
        C.seed_hi = (uint32_t)(noise_seed >> 32);
        l += launch_psf_lsf(C, P.d_cube0, P.pitch0, P.has_conv_map ? &P.conv_map : nullptr, P.d_tmp, out, st);
    }
    return l;
}

}  // namespace rubix
