// kernels.h -- internal launch interface between the C-ABI layer and the kernels.
#pragma once

#include <cuda.h>
#include <cuda_runtime.h>
#include <stddef.h>
#include <stdint.h>

#include "slab_layout.h"

namespace rubix {

struct DepRec;
struct MapRec;
struct PartRec;
struct Item;

// Streaming multiprocessors of the current device (cached per device); grid
// caps of the grid-stride kernels are multiples of it.
int sm_count();

// Deposit launch shape: threads per CTA (one CTA per SM: the SSP slab fills
// shared memory; 1024 threads leave 64 registers per thread. Mid-size and large
// galaxy, ms: 1024 threads 3.41 / 53.9, 896 3.49 / 55.9, 768 3.39 / 55.1).
#ifndef RUBIX_DEP_THREADS
#define RUBIX_DEP_THREADS 1024
#endif
// Deposit geometry: most particles per work item, the line-of-sight speed (km/s)
// the shared-memory slab's Doppler halo covers, and a fixed number of age
// bands (0 = chosen by the cost estimate).
#ifndef RUBIX_DEP_CHUNK
#define RUBIX_DEP_CHUNK 256
#endif
#ifndef RUBIX_DEP_VHALO
#define RUBIX_DEP_VHALO 800.0
#endif
#ifndef RUBIX_DEP_BANDS
#define RUBIX_DEP_BANDS 0
#endif
// Cost of a work item in particle units, for the static split of the
// (tile, item) cost space over CTAs.
#ifndef RUBIX_DEP_COSTC0
#define RUBIX_DEP_COSTC0 4
#endif
// Most work items a warp claims at once (its first lanes look them up together;
// claim_size in tile.cuh), in the deposit and in the adjoint.
#ifndef RUBIX_DEP_GRAB
#define RUBIX_DEP_GRAB 3
#endif
#ifndef RUBIX_ADJ_GRAB
#define RUBIX_ADJ_GRAB 2
#endif
// Threads of an adjoint CTA (one per SM, the deposit's slab geometry).
#ifndef RUBIX_ADJ_THREADS
#define RUBIX_ADJ_THREADS 768
#endif

// K1 parameters. The sort key is spaxel * n_bands + age band (n_bands <= 1:
// the plain spaxel key); particles outside the field get nx*ny*n_bands.
struct AssignParams {
    long long n;
    const float *x, *y, *z, *vx, *vy, *vz, *v_los;  // vx nullable (treated as 0)
    int preprojected;
    double R[9];      // orientation, row-major: x' = (R0 x + R1 y) + R2 z, ..., v_los = (R6 vx + R7 vy) + R8 vz
    double Di[3];     // dv_los/d(inclination) = Di . (vx, vy, vz)
    double Da[2];     // dv_los/d(azimuth) = Da . (vx, vy)
    float2* dv_dang;  // [n] original order (nullable): (dv_los/d inclination, dv_los/d azimuth)
    double x_lo, y_lo, inv_size;
    int nx, ny;
    int row_lo, rows; // row window: spaxel rows [row_lo, row_lo + rows) are kept (rows <= 0: all ny)
    int* key;         // [n]
    // [n] original order (nullable): (mass, age, Z, line-of-sight velocity),
    // one 16-byte record per particle, so that the setup gathers one record
    // per particle in sorted order instead of four arrays
    PartRec* pin_out;
    const float *mass, *Zm;
    // age bands (optional; the age also goes into pin_out)
    const float* age;
    const float* la_nodes;
    int n_age, apb, n_bands;
};

int launch_assign(const AssignParams& P, cudaStream_t st);
// Stable sort of keys in [0, n_keys); seg_off gets n_keys + 1 entries. scratch
// holds scratch_ints ints (sort_scratch_ints of sort_layout.h for a capacity);
// -1, with nothing launched, if the sort needs more. long_tiles: the large tiles
// whatever n is, for less scratch. Also clears next_chain (nullable), the chain of
// a scan that follows. quiet_scan (tests): the scans' blocks publish nothing.
int launch_sort_by_key(const int* keys, long long n, int n_keys, int* keys_tmp, int* vals_tmp, int* keys_out,
                       int* perm_out, int* seg_off, int* scratch, size_t scratch_ints, bool long_tiles,
                       unsigned long long* next_chain, int n_next_chain, bool quiet_scan, cudaStream_t st);

// SSP grid as seen by the kernels (the templates themselves: SlabParams).
struct SspDev {
    int dtype;              // 0 f32, 1 bf16, 2 f16
    int n_age, n_Z, n_t, n_ls;
    const float* la_nodes;  // [n_age]
    const float* lz_nodes;  // [n_Z]
    double ls0, dls;
};

// K3: per-particle setup in sorted order + work items.
struct SetupParams {
    SspDev ssp;
    const int* perm;         // sorted position -> particle index
    const int* seg_off;      // [n_s * n_bands + 2]
    int n_s, n_bands;
    const PartRec* pin;      // [n] original order: (mass, age, Z, v_los) per particle
    double l0, dl, z_cosmo, flux_scale;
    double inv_c;            // 1 / c in km/s
    double alpha_z;          // 1 / ((1 + z_cosmo) dls)
    double ls0_dls;          // ls0 / dls
    int n_lambda;
    int resample;            // 0: records map bin centres, 1: bin lower edges (bin means)
    DepRec* rec;             // [n_in]
    MapRec* map;             // [n_in]
    // the deposit's geometry: fixed-point shifts, band entries, path limits
    int fb, jc, apb, kind;
    float a_max, s_min, s_max;
    PartRec* prec;           // [n_in], for the adjoint (nullable)
    long long n_cap;         // capacity of rec / prec
};
int launch_setup(const SetupParams& P, long long n_total, cudaStream_t st);

struct ItemParams {
    const int* seg_off;      // [n_s * n_bands + 2]
    int n_s, n_bands;
    int chunk;               // max particles per item
    int* item_off;           // [n_s + 1]
    int* part_off;           // [n_s + 1]
    int* split;              // [n_s] the split spaxels, in any order
    Item* items;             // capacity item_cap
    long long item_cap;
    // item_chain_words(n_s) words, cleared (common.cuh); the last counts the
    // split spaxels
    unsigned long long* chain;
    unsigned long long* slow_count;  // nullable: the forward's count of per-bin visits, reset here
    bool quiet_scan;         // tests: the scan's blocks publish nothing
    unsigned* err;
};
size_t item_chain_words(int n_s);
int launch_items(const ItemParams& P, cudaStream_t st);

// K4: deposit. One launch deposits up to kMaxJobs galaxies (jobs) that share
// the SSP grid and the output wavelength grid.
constexpr int kMaxJobs = 64;
constexpr int kDepHeader = 1024;  // deposit shared-memory header (barrier, counters, job table)
struct DepJob {
    const DepRec* rec;
    const MapRec* map;
    const Item* items;
    const int* item_off;     // [n_s + 1]: total items at [n_s]
    const int* seg_off;      // [n_s * n_bands + 2]: in-field particles at [n_s * n_bands]
    float* cube;             // [n_s][pitch] (the first n_lambda of each row)
    float* partials;         // [part_cap][n_lambda]
    long long part_cap;
    int n_s;
    int pitch;               // cube row stride in floats (>= n_lambda)
    int resample;            // 1: bin means (records hold the bins' lower edges)
};

// Template slabs: the SSP grid's age pairs, one contiguous block per age band
// ([pad + n_ls + pad] node rows of `pitch` entries; the pad rows are zero) of
// FP32 float2 entries or, for 16-bit templates, uint32_t entries (qdt 1: BF16,
// 2: FP16). The geometry of the wavelength tiles and of their shared-memory
// slabs, shared by the deposit and the adjoint.
struct SlabParams {
    const void* pair;
    int qdt;
    long long band_stride;      // entries per band block
    int n_ls, pad, pitch, es;   // es: entries per cell index (tile.cuh)
    int n_bands;
    int band_e0[kMaxBands];     // first entry of each age band
    int kind;                   // bins per round and how lanes reach their nodes (slab_layout.h)
    int n_lambda;
    int tile_w;                 // output bins per tile = rounds x kind_bins(kind)
    int n_tiles;
    const int* tile_klo;        // [n_tiles] first SSP node of each tile's slab (a multiple of 4)
    // [2][n_tiles] node position of each tile's first bin (bin centres, then
    // lower edges) for a particle at rest, from the slab's first node, in units
    // of 2^-fb nodes
    const unsigned* tile_ref;
    int fb, jc;                 // fixed point of the records' shifts (DepRec)
    float a0_1m;                // 1 - dt/dj of a particle at rest
    float s_min, s_max;         // shifts (nodes) whose rounds stay in every tile's slab
    int slab_w;                 // nodes per slab (0 = no slab: global path only)
    float a_max;                // largest dt/dj of the fast rounds, and
    int need;                   // the nodes they read from a particle's first
    // per round of centres and of means: whole nodes, and the rest, for a
    // particle at rest
    float ib[2], fbr[2];
    const float2* lane_ref;     // [32] lane * dt/dj at rest: whole nodes, rest
    int cost_c0;                // per-item cost in particle units
    unsigned* err;
};
inline __host__ __device__ const void* band_ptr(const void* pair, int qdt, long long band_stride, int band) {
    return static_cast<const char*>(pair) + (long long)band * band_stride * (qdt ? 4 : 8);
}

// Lays the templates t ([n_age][n_Z][n_ls] FP32) out as age pairs: `pair`
// (SlabParams::pair) and, if not null, `adj`, the adjoint's FP32 entries of the
// same (storage-rounded) values: the pairs for kind 0, else (T, T(next age) - T).
int launch_build_pairs(const SlabParams& G, int apb, int n_age, int n_Z, const float* t, void* pair, float2* adj,
                       cudaStream_t st);

struct DepositParams : SlabParams {
    DepJob jobs[kMaxJobs];
    int n_jobs;
    unsigned long long* slow_count;
};
int launch_deposit(const DepositParams& P, int n_ctas, int threads, size_t smem, cudaStream_t st);
size_t deposit_smem_bytes(int pitch, int slab_w);

// Rows the deposit leaves: zeros for the spaxels without particles (no work
// item covers them; with skip_rp >= 0 only those within the fused convolution's
// reach of a particle: ConvParams::seg_off with rp = skip_rp), and the partial
// rows of split spaxels summed in a fixed order (K5): FP32 for at most
// kCombineF32Rows rows, a compensated FP32 sum (two-sum) above.
constexpr int kCombineF32Rows = 4;
struct RowParams {
    const int* seg_off;
    int nx, ny, n_bands, n_lambda, pitch, skip_rp;
    const int* part_off;
    const int* split;                    // the split spaxels
    const unsigned long long* n_split;   // their number
    long long max_split;                 // the most there can be
    const float* partials;
    float* cube;
};
int launch_rows(const RowParams& P, cudaStream_t st);

// K6: PSF + LSF (+ noise).
constexpr int kMaxRadius = 64;
struct ConvParams {
    int nx, ny, n_lambda;
    int rp, rl;                  // radii (0 = identity)
    float gp[2 * kMaxRadius + 1];
    float gl[2 * kMaxRadius + 1];
    float noise_inv_s2n;         // 0 = no noise
    uint32_t seed_lo, seed_hi;
    unsigned* err;               // device error word (bounded waits of the fused kernel; nullable)
    int ty;                      // output rows per CTA (set at launch)
    int xb_first;                // first block of kConvX columns of the launch (set at launch)
    // segment offsets of the cube's spaxels, seg_bands per spaxel (nullable): a
    // (row, block of kConvX columns) without a particle within rp columns is
    // taken as zero, unread
    const int* seg_off;
    int seg_bands;
};
constexpr int kConvX = 8;        // spaxels along x per fused CTA
// `in` rows have stride in_pitch floats; `out` is dense ([ny][nx][n_lambda]).
// in_map (nullable): a 3-D TMA map of `in` (x = wavelength over n_lambda, y = x
// spaxel, z = y spaxel; zero fill outside) over a box of conv_tma_box; without
// it `in` is dense, at any alignment.
int launch_psf_lsf(const ConvParams& P, const float* in, int in_pitch, const CUtensorMap* in_map, float* tmp,
                   float* out, cudaStream_t st);
// Box the fused kernel loads for these radii: {wavelength, x}; false if the
// radii have no fused instantiation.
bool conv_tma_box(int rp, int rl, unsigned box[2]);
// True if launch_psf_lsf needs the intermediate cube `tmp` for these radii.
bool psf_lsf_needs_tmp(int rp, int rl);

// K7/K8: adjoint.
struct AdjointParams {
    SspDev ssp;
    const PartRec* prec;       // [n_in] sorted order
    const int* perm;           // sorted position -> particle index
    const int* seg_off;        // [n_s * n_bands + 2]
    int n_s, n_bands, n_lambda;
    double l0, dl, z_cosmo, flux_scale;
    const float* G0;           // [n_s][n_lambda] dL/dcube0
    float *d_mass, *d_age, *d_Z, *d_v;   // original order, nullable
    double* contrib;           // [n_in][kGlobal] per sorted particle: dL/dv, m*dL/dm, dL/dv * dv/d(incl), dL/dv * dv/d(azim)
    const float2* dv_dang;     // [n] original order: dv_los/d(inclination), dv_los/d(azimuth)
    long long n_in;            // upper bound (grid sizing)
};

// Adjoint over the deposit's (wavelength tile, work item, age band)
// decomposition: per (tile, particle) the four sums
//   part = (sum_j G S, sum_j G dS/dta', sum_j G dS/dtz', sum_j G dS/dt * t_abs)
// over the tile's bins (unit mass), from slabs of the same geometry.
struct AdjTileParams : SlabParams {
    const MapRec* map;          // [n_in] the forward's maps (sorted order)
    const float2* wu;           // [n_in] position (ta, tz) in the SSP cell
    const Item* items;
    const int* item_off;        // [n_s + 1]
    const int* seg_off;         // [n_s * n_bands + 2]
    int n_s;
    const float* G0;            // [n_s][n_lambda] dL/d(cube before PSF/LSF)
    float4* part;               // [n_tiles][n_cap]
    long long n_cap;
    float ls0_over;             // ls0 / dls: node index -> rest wavelength / dls
    int resample;               // 1: bin means (records hold the bins' lower edges)
};
int launch_adjoint_tiles(const AdjTileParams& P, int n_ctas, int threads, size_t smem, cudaStream_t st);
// Position in the SSP cell per sorted particle (K7 setup).
int launch_adjoint_setup(const AdjointParams& P, float2* wu, cudaStream_t st);
// Sum of the tiles' parts in FP64 (tile order) and the chain rule to
// dL/d(mass, age, Z, v_los) in original order (+ contributions to global sums).
int launch_adjoint_final(const AdjointParams& P, const float4* part, int n_tiles, long long n_cap, cudaStream_t st);
int launch_zero_grads(float* a, float* b, float* c, float* d, long long n, cudaStream_t st);
// Gradients of the shared parameters: dL/dv_sys, dL/dln(M), dL/d(inclination), dL/d(azimuth).
constexpr int kGlobal = 4;
int launch_reduce_global(const double* contrib, const int* n_in_dev, double* out, double* scratch, cudaStream_t st);

}  // namespace rubix
