// rows.cu -- the cube rows the deposit does not write itself (the per-spaxel
// sum of Sec. 3): rows of spaxels without particles, and rows of split
// spaxels, summed from their work items' partial rows.
#include "common.cuh"
#include "conv_layout.h"
#include "kernels.h"
#include "twosum.cuh"

namespace rubix {

// ----------------------------------------------------------------------------
// Rows of spaxels without particles: zeros (one warp per row, 16-byte stores
// when the rows are 16-byte aligned). The deposit has no work item for them,
// so a small galaxy in a large field costs the deposit only its own spaxels.
// Before a convolution, rows out of reach of any particle are left alone: the
// fused PSF/LSF kernel takes (row, block of columns) pairs without a particle
// in reach as zero without reading them (1e4 particles in 300 x 300 x 3721:
// zero rows 0.21 ms and PSF/LSF 0.75 ms when all are written and read).
// ----------------------------------------------------------------------------
__device__ __forceinline__ void zero_rows(const RowParams& P, long long w0, long long nw, int lane) {
    const int nb = P.n_bands, nx = P.nx;
    const long long n_s = (long long)nx * P.ny;
    const bool vec = (P.pitch % 4) == 0 && (reinterpret_cast<uintptr_t>(P.cube) & 15) == 0;
    for (long long s = w0; s < n_s; s += nw) {
        if (P.seg_off[(s + 1) * nb] != P.seg_off[s * nb]) continue;
        if (P.skip_rp >= 0) {
            // is it read: by a block whose columns, widened by rp, hold both the
            // spaxel and a particle of its row
            const long long y = s / nx;
            const int x = (int)(s - y * nx), rp = P.skip_rp;
            const int* row = P.seg_off + y * nx * nb;
            bool read = false;
            for (int b = max(x - rp, 0) / kConvX; b <= (x + rp) / kConvX && b * kConvX < nx; ++b)
                read = read || row[min((b + 1) * kConvX + rp, nx) * nb] != row[max(b * kConvX - rp, 0) * nb];
            if (!read) continue;
        }
        float* row = P.cube + s * P.pitch;
        int j0 = 0;
        if (vec) {
            float4* r4 = reinterpret_cast<float4*>(row);
            const int n4 = P.n_lambda >> 2;
            for (int j = lane; j < n4; j += 32) r4[j] = make_float4(0.f, 0.f, 0.f, 0.f);
            j0 = n4 << 2;
        }
        for (int j = j0 + lane; j < P.n_lambda; j += 32) row[j] = 0.f;
    }
}

// ----------------------------------------------------------------------------
// K5: rows of split spaxels = the sum of their partial rows in item order: a
// plain FP32 sum for spaxels of at most kCombineF32Rows items, a compensated
// FP32 sum above (very high-count spaxels). The compensated sum carries the
// rounding error of every addition (Knuth's two-sum: s + e is exactly the
// sum of s and x) in a second FP32 accumulator: the error before the final
// rounding stays within about n^2 2^-48 of the rows' magnitudes, far below
// one FP32 rounding, as with an FP64 accumulator, without the FP64 pipe,
// which on this GPU runs at 1/64 of the FP32 rate.
// ----------------------------------------------------------------------------

// One unit = kCombineBins bins of one split spaxel's row, taken by one warp
// (lane l sums bins l, l + 32, l + 64, l + 96 of the unit: four independent
// loads per partial row in flight), so that the rows of a very high-count
// spaxel are summed by many warps at once and each warp has several loads
// in flight while it waits on the next unit's row offsets.
__device__ __forceinline__ void combine_rows(const RowParams& P, long long warp, long long n_warps, int lane) {
    const int n_split = (int)*P.n_split, n_lambda = P.n_lambda;
    const int n_chunks = (n_lambda + kCombineBins - 1) / kCombineBins;
    const long long n_units = (long long)n_split * n_chunks;
    for (long long u = warp; u < n_units; u += n_warps) {
        const int s = P.split[u / n_chunks];
        const int j0 = (int)(u % n_chunks) * kCombineBins + lane;
        const int p0 = P.part_off[s], nr = P.part_off[s + 1] - p0;
        const float* __restrict__ col = P.partials + (long long)p0 * n_lambda;
        float acc[4] = {0.f, 0.f, 0.f, 0.f}, err[4] = {0.f, 0.f, 0.f, 0.f};
        bool in[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) in[k] = j0 + 32 * k < n_lambda;
        if (nr <= kCombineF32Rows) {
            // a few partial rows: FP32 adds lose nothing that the FP32 partial
            // sums have not already lost
            for (int r = 0; r < nr; ++r)
#pragma unroll
                for (int k = 0; k < 4; ++k)
                    if (in[k]) acc[k] += col[(long long)r * n_lambda + j0 + 32 * k];
        } else {
#pragma unroll 2
            for (int r = 0; r < nr; ++r)
#pragma unroll
                for (int k = 0; k < 4; ++k)
                    if (in[k]) two_sum_add(acc[k], err[k], col[(long long)r * n_lambda + j0 + 32 * k]);
#pragma unroll
            for (int k = 0; k < 4; ++k) acc[k] += err[k];
        }
#pragma unroll
        for (int k = 0; k < 4; ++k)
            if (in[k]) P.cube[(long long)s * P.pitch + j0 + 32 * k] = acc[k];
    }
}

// The split spaxels' rows first: they take longest.
__global__ void __launch_bounds__(kRowThreads) k_rows(const __grid_constant__ RowParams P) {
    const int lane = threadIdx.x & 31;
    const long long warp = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const long long n_warps = ((long long)gridDim.x * blockDim.x) >> 5;
    combine_rows(P, warp, n_warps, lane);
    zero_rows(P, warp, n_warps, lane);
}

int launch_rows(const RowParams& P, cudaStream_t st) {
    const long long n_s = (long long)P.nx * P.ny;
    if (n_s < 1) return 0;
    k_rows<<<row_blocks(n_s, P.max_split, P.n_lambda, sm_count()), kRowThreads, 0, st>>>(P);
    return 1;
}

}  // namespace rubix
