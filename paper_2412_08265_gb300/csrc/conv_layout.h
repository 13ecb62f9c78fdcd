// conv_layout.h -- output rows per CTA of the fused PSF/LSF kernel (psf_lsf.cu):
// host arithmetic without a GPU.
#pragma once

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

}  // namespace rubix
