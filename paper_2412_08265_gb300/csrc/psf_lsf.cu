// psf_lsf.cu -- observational effects (Sec. 3: the cube is convolved with the
// instrument's point-spread and line-spread functions and noise is added;
// Sec. 4: both functions are Gaussian).
//
// The 3-D kernel is separable, g(dy) g(dx) h(dj), with zero padding on every
// axis. For the radii of the instruments used here a single fused pass
// (k_psf_lsf, below) reads the cube once and writes it once. Other radii
// take two passes through an intermediate cube:
//   pass 1 (k_lsf_psfx): one CTA per (wavelength chunk, x chunk, row y) loads
//     the row segment with its halos into shared memory, applies the LSF along
//     wavelength and then the PSF along x, and writes an intermediate cube;
//   pass 2 (k_psfy_noise): each thread owns one (x, wavelength) column of a
//     y-chunk and applies the PSF along y, then optional Philox noise.
// All global accesses run along wavelength (the fastest axis): coalesced.
#include <algorithm>

#include "common.cuh"
#include "conv_layout.h"
#include "kernels.h"

namespace rubix {

constexpr int kLC = 64;   // wavelength bins per CTA in pass 1
constexpr int kXC = 64;   // spaxels along x per CTA in pass 1

__global__ void __launch_bounds__(256) k_lsf_psfx(const ConvParams P, const float* __restrict__ in,
                                                  float* __restrict__ out) {
    extern __shared__ float sm[];
    const int rl = P.rl, rp = P.rp;
    const int W_in = kLC + 2 * rl;
    const int XW = kXC + 2 * rp;
    float* s_in = sm;                  // [XW][W_in]
    float* s_mid = sm + XW * W_in;     // [XW][kLC]
    const int j0 = blockIdx.x * kLC;
    const int x0 = blockIdx.y * kXC;
    const int y = blockIdx.z;
    const int nx = P.nx, nl = P.n_lambda;
    const long long row = (long long)y * nx;
    for (int e = threadIdx.x; e < XW * W_in; e += blockDim.x) {
        const int xi = e / W_in, l = e - xi * W_in;
        const int x = x0 - rp + xi, j = j0 - rl + l;
        s_in[e] = (x >= 0 && x < nx && j >= 0 && j < nl) ? in[(row + x) * nl + j] : 0.f;
    }
    __syncthreads();
    for (int e = threadIdx.x; e < XW * kLC; e += blockDim.x) {
        const int xi = e / kLC, l = e - xi * kLC;
        const float* src = s_in + xi * W_in + l;
        float acc = 0.f;
        for (int d = 0; d <= 2 * rl; ++d) acc = fmaf(P.gl[d], src[d], acc);
        s_mid[e] = acc;
    }
    __syncthreads();
    for (int e = threadIdx.x; e < kXC * kLC; e += blockDim.x) {
        const int xi = e / kLC, l = e - xi * kLC;
        const int x = x0 + xi, j = j0 + l;
        if (x >= nx || j >= nl) continue;
        const float* src = s_mid + xi * kLC + l;
        float acc = 0.f;
        for (int d = 0; d <= 2 * rp; ++d) acc = fmaf(P.gp[d], src[d * kLC], acc);
        out[(row + x) * nl + j] = acc;
    }
}

__device__ __forceinline__ float add_noise(float v, long long idx, float inv_s2n, uint32_t seed_lo, uint32_t seed_hi) {
    U4 c;
    c.x = (uint32_t)idx;
    c.y = (uint32_t)((unsigned long long)idx >> 32);
    c.z = 0u;
    c.w = 0u;
    const U4 r = philox4x32_10(c, seed_lo, seed_hi);
    const float u1 = (float)((r.x >> 8) + 1u) * (1.0f / 16777216.0f);  // (0, 1]
    const float u2 = (float)(r.y >> 8) * (1.0f / 16777216.0f);         // [0, 1)
    const float z = sqrtf(-2.0f * logf(u1)) * cospif(2.0f * u2);
    return fmaf(fabsf(v) * inv_s2n, z, v);
}

// The same for 4 voxels, out of line: the fused kernel's unrolled rows would
// hold 28 copies, and their length costs instruction fetches.
__device__ __noinline__ float4 add_noise4(float4 v, long long idx, float inv_s2n, uint32_t seed_lo, uint32_t seed_hi) {
    return make_float4(add_noise(v.x, idx, inv_s2n, seed_lo, seed_hi), add_noise(v.y, idx + 1, inv_s2n, seed_lo, seed_hi),
                       add_noise(v.z, idx + 2, inv_s2n, seed_lo, seed_hi),
                       add_noise(v.w, idx + 3, inv_s2n, seed_lo, seed_hi));
}

constexpr int kYC = 32;  // rows per thread in pass 2

__global__ void __launch_bounds__(256) k_psfy_noise(const ConvParams P, const float* __restrict__ in,
                                                    float* __restrict__ out) {
    const long long plane = (long long)P.nx * P.n_lambda;  // one y row of the cube
    const long long col = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (col >= plane) return;
    const int y0 = blockIdx.y * kYC;
    const int y1 = min(y0 + kYC, P.ny);
    const int rp = P.rp;
    for (int y = y0; y < y1; ++y) {
        float acc = 0.f;
        for (int d = -rp; d <= rp; ++d) {
            const int yy = y + d;
            if (yy < 0 || yy >= P.ny) continue;
            acc = fmaf(P.gp[d + rp], in[(long long)yy * plane + col], acc);
        }
        const long long idx = (long long)y * plane + col;
        if (P.noise_inv_s2n > 0.f) acc = add_noise(acc, idx, P.noise_inv_s2n, P.seed_lo, P.seed_hi);
        out[idx] = acc;
    }
}


// ----------------------------------------------------------------------------
// Fused single pass for the common radii (compile-time rp, rl): the cube is
// read once (plus halos) and written once. One CTA owns kTX = 8 spaxels along
// x (one per warp) x ty rows along y x kTL = kTB - 2 RLa bins. Each input row
// (kTB = 128 bins from j0 - RLa, spaxels x0 - rp .. x0 + kTX + rp) arrives by
// asynchronous copies in a kTS-stage mbarrier ring:
//   pitched rows (the deposit's own cube, 16-byte rows): one 3-D TMA box, whose
//     zero fill outside the cube is the zero padding;
//   dense rows of any alignment (a caller's cube): one bulk copy per spaxel of
//     the 16-byte granules that hold its bins (DenseRows).
//   PSF along x: each warp takes four output columns over 32 bins, one bin per
//     lane: 4 + 2 rp conflict-free 4-byte loads (at any row alignment) for four
//     outputs; with one column and four bins per lane it was 2 rp + 1 16-byte
//     loads, nearly three times the shared-memory wavefronts, which bound the
//     kernel. Into px, every bin the LSF needs, halo included.
//   LSF along wavelength: warp w owns output column x0 + w, lane q bins 4q ..
//     4q + 3 of its px row (lanes RLa/4 .. 31 - RLa/4, the tile's). Then the PSF-y
//     register accumulators: the value of input row y_in is added, with weight
//     gp[m], to the accumulator of output row y_in - rp + m (2 rp + 1 per owned
//     bin, each moved down one place by the same multiply-add), and the output
//     row y_in - rp is then complete: noise is added and it is written once.
// One CTA barrier per input row (every warp is done with the stage before it
// is refilled, and px is complete; a barrier per two or three rows measured no
// faster). The terms of each output are summed
// in the same order for both forms (PSF x, LSF, PSF y; each over its taps in
// order), so they give the same bits.
//
// Bound by instruction issue (75 % of the slots; shared-memory wavefronts 67 %) and
// the barrier per row: 150 x 150 spaxels x 3721 bins in 164 us, the dense form 81 x
// 150 x 3721 in 127 us = 0.42 of the copy bandwidth (a kernel of 4-byte cp.async
// copies took 323 us).
// ----------------------------------------------------------------------------
#ifndef RUBIX_PSF_TSTAGES
#define RUBIX_PSF_TSTAGES 4
#endif
#ifndef RUBIX_PSF_TMINB
#define RUBIX_PSF_TMINB 4       // CTAs per SM the register budget is sized for
#endif
constexpr int kTB = 128, kTX = kConvX, kTThreads = 256, kTWarps = kTThreads / 32;
constexpr int kTS = RUBIX_PSF_TSTAGES;
constexpr int kHead = 64;              // header, in floats: mbarriers, then the row bits
static_assert(kTX == kTWarps, "one output column per warp");
static_assert(kTS * 8 <= 128, "mbarriers before the row bits");

template <int RP, int RL, bool DENSE = false>
struct TmaGeo {
    static constexpr int RLa = (RL + 3) / 4 * 4;  // wavelength halo rounded up to 16 bytes
    static constexpr int LW = kTB;                // box: bins
    static constexpr int TL = kTB - 2 * RLa;      // output bins per tile
    static constexpr int XW = kTX + 2 * RP;       // box: spaxels along x
    static constexpr int NV = 1 + RLa / 2;        // 16-byte loads per lane for 4 LSF outputs
    static constexpr int row = LW + (DENSE ? 4 : 0);  // stage row: dense rows start anywhere in a 16-byte granule
    static constexpr int stage_floats = (row * XW + 31) / 32 * 32;  // stages stay 128-byte aligned
    static constexpr size_t smem = 4 * kHead + (size_t)kTS * stage_floats * 4 + (size_t)2 * kTX * kTB * 4;
};

// Dense input rows: float cube [ny][nx][nl] at any 4-byte aligned address.
// `al` is that address rounded down to 16 bytes, `off` (0..3) the floats
// between; positions count floats from `al`. Copies take whole 16-byte granules
// that hold at least one float of the cube, except the last, partial one (its
// end may lie past the buffer): those floats are read and stored singly.
struct DenseRows {
    const float* al;
    long long off, full;  // first position of the cube; end of its whole granules
};

template <int RP, int RL, bool DENSE, bool NOISE>
__global__ void __launch_bounds__(kTThreads, RUBIX_PSF_TMINB) k_psf_lsf(const __grid_constant__ ConvParams P,
                                                                       const __grid_constant__ CUtensorMap in_map,
                                                                       const DenseRows D, float* __restrict__ out) {
    using G = TmaGeo<RP, RL, DENSE>;
    constexpr int NR = 2 * RP + 1;
    constexpr int Q0 = G::RLa / 4, Q1 = 32 - G::RLa / 4;  // lanes whose bins are the tile's
    extern __shared__ __align__(1024) float smt[];
    uint64_t* bars = reinterpret_cast<uint64_t*>(smt);
    float* stages = smt + kHead;
    float* px = stages + kTS * G::stage_floats;  // [2][kTX][kTB] PSF-x output, alternating by row
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int j0 = blockIdx.x * G::TL, x0 = (int)(P.xb_first + blockIdx.y) * kTX, y0 = blockIdx.z * P.ty;
    const int y1 = min(y0 + P.ty, P.ny);
    const int nx = P.nx, nl = P.n_lambda;
    const int n_rows = (y1 - y0) + 2 * RP;  // input rows y0 - RP .. y1 + RP - 1
    float gl[2 * RL + 1], gp[NR];
#pragma unroll
    for (int d = 0; d <= 2 * RL; ++d) gl[d] = P.gl[d];
#pragma unroll
    for (int d = 0; d < NR; ++d) gp[d] = P.gp[d];
    if (threadIdx.x == 0) {
        // arrivals per phase: the one box, or each copied column's lane
        const int n = DENSE ? min(x0 + kTX + RP, nx) - max(x0 - RP, 0) : 1;
        for (int s = 0; s < kTS; ++s) mbar_init(&bars[s], n);
        fence_mbar_init();
    }
    // which input rows hold anything for this CTA: rows outside the cube, or
    // without a particle within reach of these columns, are zero
    unsigned* s_live = reinterpret_cast<unsigned*>(smt) + 32;
    for (int i0 = warp * 32; i0 < n_rows; i0 += kTThreads) {
        const int y = y0 - RP + i0 + lane;
        const bool on = i0 + lane < n_rows && y >= 0 && y < P.ny &&
                        (!P.seg_off || P.seg_off[((long long)y * nx + min(x0 + kTX + RP, nx)) * P.seg_bands] !=
                                           P.seg_off[((long long)y * nx + max(x0 - RP, 0)) * P.seg_bands]);
        const unsigned m = __ballot_sync(0xffffffffu, on);
        if (lane == 0) s_live[i0 >> 5] = m;
    }
    if constexpr (DENSE) {
        // columns outside the cube are zero in every stage and never copied
        for (int c = warp; c < G::XW; c += kTWarps)
            if (x0 - RP + c < 0 || x0 - RP + c >= nx)
                for (int k = lane; k < kTS * G::row; k += 32)
                    stages[k / G::row * G::stage_floats + c * G::row + k % G::row] = 0.f;
    }
    __syncthreads();
    auto live = [&](int i) { return (s_live[i >> 5] >> (i & 31)) & 1u; };
    // dense rows: the lane's spaxel column (warp 0), whose granules of bins
    // [j_a, j_b) it copies
    const bool copies = lane < G::XW && x0 - RP + lane >= 0 && x0 - RP + lane < nx;
    const int j_a = max(j0 - G::RLa, 0), j_b = min(j0 - G::RLa + G::LW, nl);
    const long long row_len = (long long)nx * nl;
    const long long row0 = D.off + (long long)(y0 - RP) * row_len + (long long)(x0 - RP + lane) * nl;
    auto issue = [&](int i, int s) {  // input row i into stage s (warp 0)
        if constexpr (!DENSE) {
            if (lane == 0) {
                fence_proxy_async_smem();
                mbar_arrive_expect_tx(&bars[s], (uint32_t)(G::LW * G::XW * 4));
                tma_load_3d(stages + s * G::stage_floats, &in_map, &bars[s], j0 - G::RLa, x0 - RP, y0 - RP + i);
            }
        } else {
            // lane xi copies the granules of spaxel x0 - RP + xi's bins
            if (copies) {
                const long long row = row0 + i * row_len;
                const long long a4 = (row + j_a) & ~3ll;
                const uint32_t bytes = (uint32_t)max(min((row + j_b + 3) & ~3ll, D.full) - a4, 0ll) * 4u;
                float* dst = stages + s * G::stage_floats + lane * G::row;
                // position of the stage row's first float: (row + j0 - RLa) & ~3
                const int at = (int)(a4 - ((row + j0 - G::RLa) & ~3ll));
                // the cube's last, partial granule
                for (long long e = max(a4, D.full); e < row + j_b; ++e) dst[at + (int)(e - a4)] = D.al[e];
                fence_proxy_async_smem();
                mbar_arrive_expect_tx(&bars[s], bytes);
                if (bytes) bulk_load(smem_addr(dst + at), D.al + a4, bytes, &bars[s]);
            }
        }
    };
    // rows that hold nothing take no stage; live rows take the stages in turn
    int next = 0, issued = 0;  // warp 0: next input row to look at, live rows issued
    auto issue_next = [&]() {
        while (next < n_rows && !live(next)) ++next;
        if (next < n_rows) {
            issue(next, issued % kTS);
            ++next;
            ++issued;
        }
    };
    if (warp == 0)
        for (int k = 0; k < kTS; ++k) issue_next();
    int turn = 0;  // live rows taken

    float2 acc[NR][2];
#pragma unroll
    for (int m = 0; m < NR; ++m) acc[m][0] = acc[m][1] = make_float2(0.f, 0.f);
    const float* prow = px;  // column warp's row of the current px buffer
    // PSF-x: the warp's first column of the tile and the lane's bin of the box
    const int c0 = (warp & 1) * 4, xb = (warp >> 1) * 32 + lane;
    const bool owns = lane >= Q0 && lane < Q1;
    const int x = x0 + warp;
    const int jl = j0 - G::RLa + 4 * lane;  // cube bin of the lane's first box bin
    // dense rows: position (modulo 2^32) of input column c0's first bin in input row 0
    const unsigned row_step = (unsigned)nx * (unsigned)nl;
    const unsigned col0 = (unsigned)D.off + (unsigned)(y0 - RP) * row_step + (unsigned)(x0 - RP + c0) * (unsigned)nl + (unsigned)(j0 - G::RLa);

    // rows of `out` that are 16-byte aligned take 16-byte stores (others four
    // 4-byte ones: bringing them into order through shared memory first cost more
    // than it saved)
    const bool vec = (nl & 3) == 0 && (reinterpret_cast<uintptr_t>(out) & 15) == 0;

    float* orow = out + ((long long)(y0 - 2 * RP) * nx + x) * nl + j0 - G::RLa;  // of the row input row i completes
    const long long ostep = (long long)nx * nl;
    unsigned bits = 0;
    for (int i = 0; i < n_rows; ++i, orow += ostep, bits >>= 1) {
        if ((i & 31) == 0) bits = s_live[i >> 5];
        const bool has = bits & 1u;  // uniform over the CTA
        if (has) {
            const int s = turn % kTS;
            const bool ok = mbar_wait_bounded(&bars[s], (uint32_t)((turn / kTS) & 1), 2000000000ll);
            float* pbuf = px + (turn & 1) * kTX * kTB;
            if (ok) {
                // PSF along x: 4 output columns from 4 + 2 RP input columns, one bin per lane
                const float* src = stages + s * G::stage_floats + c0 * G::row + xb;
                float c[4 + 2 * RP];
                const unsigned p = col0 + (unsigned)i * row_step;  // DENSE: position of column c0's row
#pragma unroll
                for (int d = 0; d < 4 + 2 * RP; ++d)
                    c[d] = src[d * G::row + (DENSE ? (int)((p + (unsigned)(d * nl)) & 3u) : 0)];
                const bool in = !DENSE || (j0 - G::RLa + xb >= 0 && j0 - G::RLa + xb < nl);
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    float a = 0.f;
#pragma unroll
                    for (int d = 0; d < NR; ++d) a = fmaf(gp[d], c[q + d], a);
                    pbuf[(c0 + q) * kTB + xb] = in ? a : 0.f;
                }
            }
            if (__syncthreads_or(!ok)) {
                // a load did not complete in time: record it, let the copies in
                // flight land (bounded), and stop
                if (threadIdx.x == 0) {
                    if (P.err) atomicOr(P.err, kErrTmaTimeout);
                    for (int r = turn; r < issued; ++r)
                        mbar_wait_bounded(&bars[r % kTS], (uint32_t)((r / kTS) & 1), 200000000ll);
                }
                return;
            }
            // every warp is done with stage s: refill it. The barrier also made
            // the px rows visible; they alternate, so that the next row's are not
            // written before every warp has read these
            prow = pbuf + warp * kTB;
            ++turn;
            if (warp == 0) issue_next();
        }
        float o[4] = {0.f, 0.f, 0.f, 0.f};
        if (has && owns) {
            // LSF along wavelength from px: bins 4 lane - RLa .. 4 lane + 3 + RLa
            const float4* r4 = reinterpret_cast<const float4*>(prow + 4 * lane - G::RLa);
            float v[4 * G::NV];
#pragma unroll
            for (int c = 0; c < G::NV; ++c) {
                const float4 t = r4[c];
                v[4 * c] = t.x;
                v[4 * c + 1] = t.y;
                v[4 * c + 2] = t.z;
                v[4 * c + 3] = t.w;
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                float b = 0.f;
#pragma unroll
                for (int d = 0; d <= 2 * RL; ++d) b = fmaf(gl[d], v[u + d + G::RLa - RL], b);
                o[u] = b;
            }
        }
        // acc[m] holds output row y_in - RP + m - 1 until this row's share moves it
        // down by one: no rotation, so the loop stays short (unrolled by 2 rp + 1
        // rows it waited on instruction fetches)
        const float2 o01 = make_float2(o[0], o[1]), o23 = make_float2(o[2], o[3]);
#pragma unroll
        for (int m = 0; m < NR; ++m) {
            const float2 g2 = make_float2(gp[m], gp[m]);
            acc[m][0] = __ffma2_rn(g2, o01, m + 1 < NR ? acc[m + 1][0] : make_float2(0.f, 0.f));
            acc[m][1] = __ffma2_rn(g2, o23, m + 1 < NR ? acc[m + 1][1] : make_float2(0.f, 0.f));
        }
        const int y_done = y0 + i - 2 * RP;  // output row completed by this input row
        const bool write = y_done >= y0 && x < nx;
        float4 v = make_float4(acc[0][0].x, acc[0][0].y, acc[0][1].x, acc[0][1].y);
        if constexpr (NOISE) {
            if (write && owns)
                v = add_noise4(v, ((long long)y_done * nx + x) * nl + jl, P.noise_inv_s2n, P.seed_lo, P.seed_hi);
        }
        if (write && owns) {
            if (vec) {
                if (jl < nl) *reinterpret_cast<float4*>(orow + 4 * lane) = v;
            } else {
                if (jl < nl) orow[4 * lane] = v.x;
                if (jl + 1 < nl) orow[4 * lane + 1] = v.y;
                if (jl + 2 < nl) orow[4 * lane + 2] = v.z;
                if (jl + 3 < nl) orow[4 * lane + 3] = v.w;
            }
        }
    }
}

// Radii with a fused instantiation: the PSF of FWHM 1.5 spaxels (rp = 3) and
// LSFs of sigma 1.2 A on 1.25 A or 3 A bins (rl = 4, 2), plus neighbours (the
// wavelength halo of at most 8 bins).
#define RUBIX_TMA_RADII(X) X(3, 4) X(3, 2) X(3, 0) X(0, 4) X(0, 2) X(2, 4) X(4, 4) X(3, 3) X(3, 5)

bool conv_tma_box(int rp, int rl, unsigned box[2]) {
#define RUBIX_TMA_BOX(RP_, RL_)                    \
    if (rp == RP_ && rl == RL_) {                  \
        box[0] = (unsigned)TmaGeo<RP_, RL_>::LW;   \
        box[1] = (unsigned)TmaGeo<RP_, RL_>::XW;   \
        return true;                               \
    }
    RUBIX_TMA_RADII(RUBIX_TMA_BOX)
#undef RUBIX_TMA_BOX
    return false;
}

constexpr int kMaxTY = 600;  // input rows (ty + 2 rp) have a bit each in the kernel's header

template <int RP, int RL, bool DENSE, bool NOISE>
static bool launch_conv(ConvParams P, const CUtensorMap* map, const DenseRows& D, float* out, cudaStream_t st) {
    using G = TmaGeo<RP, RL, DENSE>;
    static_assert(G::smem <= 200 * 1024, "PSF/LSF tile does not fit shared memory");
    // per launch: the attribute belongs to the current device
    if (cudaFuncSetAttribute(k_psf_lsf<RP, RL, DENSE, NOISE>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)G::smem) !=
        cudaSuccess)
        return false;
    const int n_lt = (P.n_lambda + G::TL - 1) / G::TL, n_xb = (P.nx + kTX - 1) / kTX;
    P.ty = rows_per_cta(P.ny, RP, (long long)n_lt * n_xb, (long long)RUBIX_PSF_TMINB * sm_count(), kMaxTY);
    // grid.y ends at 65535: a field of more than 524,280 spaxels along x (up to 2^24)
    // takes several launches. (Column blocks in grid.x, whose end is far off, with
    // the wavelength tiles in grid.y: 1e4 particles in 300 x 300 x 3721, 600 -> 726
    // us; both in grid.x by a division: the convolution of 81 x 150 x 3721, 127 -> 133;
    // a first column that is not known as a multiple of 8: 131.)
    for (int b = 0; b < n_xb; b += 65535) {
        P.xb_first = b;
        const dim3 g(n_lt, std::min(n_xb - b, 65535), (P.ny + P.ty - 1) / P.ty);
        k_psf_lsf<RP, RL, DENSE, NOISE><<<g, kTThreads, G::smem, st>>>(P, *map, D, out);
    }
    return true;
}

static bool try_conv(const ConvParams& P, const CUtensorMap* map, const float* in, float* out, cudaStream_t st) {
    DenseRows D{};
    const uintptr_t a = reinterpret_cast<uintptr_t>(in);
    D.al = reinterpret_cast<const float*>(a & ~(uintptr_t)15);
    D.off = (long long)((a & 15) / sizeof(float));
    D.full = (D.off + (long long)P.ny * P.nx * P.n_lambda) & ~3ll;
    const CUtensorMap none{};
    const bool noise = P.noise_inv_s2n > 0.f;
    if (noise && !map) return false;  // (no caller asks for it)
#define RUBIX_CONV_CASE(RP_, RL_)                                                                       \
    if (P.rp == RP_ && P.rl == RL_)                                                                      \
        return !map ? launch_conv<RP_, RL_, true, false>(P, &none, D, out, st)                           \
                    : (noise ? launch_conv<RP_, RL_, false, true>(P, map, D, out, st)                    \
                             : launch_conv<RP_, RL_, false, false>(P, map, D, out, st));
    RUBIX_TMA_RADII(RUBIX_CONV_CASE)
#undef RUBIX_CONV_CASE
    return false;
}

bool psf_lsf_needs_tmp(int rp, int rl) {
    unsigned box[2];
    return !conv_tma_box(rp, rl, box);
}

int launch_psf_lsf(const ConvParams& P, const float* in, int in_pitch, const CUtensorMap* in_map, float* tmp,
                   float* out, cudaStream_t st) {
    if (!in_map && in_pitch != P.n_lambda) return -1;  // without a map: dense rows
    if (try_conv(P, in_map, in, out, st)) return 1;  // (wide fields: a few launches, counted as one)
    // generic radii: two passes through an intermediate cube
    const int XW = kXC + 2 * P.rp;
    const size_t smem = (size_t)XW * (kLC + 2 * P.rl + kLC) * sizeof(float);
    cudaFuncSetAttribute(k_lsf_psfx, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
    dim3 g1((P.n_lambda + kLC - 1) / kLC, (P.nx + kXC - 1) / kXC, P.ny);
    k_lsf_psfx<<<g1, 256, smem, st>>>(P, in, tmp);
    const long long plane = (long long)P.nx * P.n_lambda;
    dim3 g2((unsigned)((plane + 255) / 256), (P.ny + kYC - 1) / kYC);
    k_psfy_noise<<<g2, 256, 0, st>>>(P, tmp, out);
    return 2;
}

}  // namespace rubix
