// conv_layout.h -- grids of the passes after the deposit, as host arithmetic
// without a GPU: blocks of the row pass (rows.cu), output rows per CTA of the fused
// PSF/LSF kernel (psf_lsf.cu).
#pragma once

#include <algorithm>

namespace rubix {

// The split of ny rows that fills whole waves of the `slots` resident CTAs with
// the fewest input rows (each CTA reads 2 rp rows more than it writes), for
// `columns` CTAs per split; at most max_ty rows. One wave of 150-row CTAs is best
// for 150 x 150 spaxels x 3721 bins; a 25 x 25 x 1000 cube runs 36 CTAs unsplit.
// *tried (nullable) counts the splits looked at.
inline int rows_per_cta(int ny, int rp, long long columns, long long slots, int max_ty, int* tried = nullptr) {
    int best = ny;
    double cost = 1e300;
    // each height ceil(ny / k) once, from the largest allowed: a radius of 0 never
    // leaves the loop early, and ny counts up to 2^24
    int ty = 0;
    for (int k = (ny + max_ty - 1) / max_ty; k <= ny; k = ty > 1 ? (ny + ty - 2) / (ty - 1) : ny + 1) {
        ty = (ny + k - 1) / k;
        if (tried) ++*tried;
        if (ty < 2 * rp && best <= max_ty) break;
        const long long ctas = columns * ((ny + ty - 1) / ty);
        // the rows of the CTAs one slot takes, and a pipeline start for each
        const double c = (double)((ctas + slots - 1) / slots) * (ty + 2 * rp + 4);
        if (c < cost * 0.999) {
            cost = c;
            best = ty;
        }
    }
    return best;
}

constexpr int kRowThreads = 256;
constexpr int kCombineBins = 128;  // bins of one row per combine unit: 4 per lane of one warp

// Blocks of the row pass: a warp per spaxel (zero rows) or per combine unit (rows of
// at most max_split split spaxels), up to eight blocks per SM.
inline int row_blocks(long long n_s, long long max_split, int n_lambda, int n_sm) {
    const long long units = std::min(max_split, n_s) * ((n_lambda + kCombineBins - 1) / kCombineBins);
    const long long warps = std::max(n_s, units), per = kRowThreads / 32;
    return (int)std::min((warps + per - 1) / per, 8ll * n_sm);
}

}  // namespace rubix
