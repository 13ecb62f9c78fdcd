// slab_layout.h -- wavelength tiles, age bands and template slabs of the deposit and
// the adjoint, and the fixed point of the particles' Doppler shifts: host arithmetic
// without a GPU.
#pragma once

#include <algorithm>
#include <cmath>
#include <vector>

namespace rubix {

constexpr int kMaxBands = 32;

// Rounds per wavelength tile that the deposit and the adjoint are built for.
#define RUBIX_ROUNDS(X) X(1) X(2) X(3) X(4) X(6) X(8) X(10) X(11) X(12)

// Geometry of the rounds: a warp takes a particle's tile in rounds of kBins
// consecutive bins, lane l owning bin j0 + kBins r + l. The kind follows from
// the bin step in template nodes A = dt/dj (chosen once per wavelength grid):
//   0: A near 1 (1 - A in [0, 1/31)): 31 bins, lanes on consecutive nodes;
//   1: A in [1/2, 1): 30 bins, each lane on its bin's node, the next node's
//      value from lane l + 1 or l + 2;
//   2: any A: 32 bins, each lane reads both of its bin's nodes; at bin centres, for
//      A in (1.03, 1.95) and CTAs with many work items, lanes read consecutive nodes
//      instead and each bin takes its two from them by shuffles (rounds_gather).
constexpr int kind_bins(int kind) { return kind == 0 ? 31 : kind == 1 ? 30 : 32; }

struct SlabLayout {
    int kind, rounds, tile_w, n_tiles;
    int apb, n_bands, nzc;      // age cells per band; bands; entries per age cell and node
    int pitch;                  // entries per node, odd
    int slab_w;                 // nodes per slab (a multiple of 4; 0 = no slab)
    int last, need;             // last bin of a tile that rounds touch; nodes they read from a particle's first
    float a_max;                // steepest dt/dj whose rounds stay within `need`
    float ib[2], fbr[2], a0_1m;
    int fb, jc;                 // fixed point of the shifts: bits after the point, bin they are taken at
    float s_min, s_max;         // shifts (nodes) whose rounds stay in every tile's slab
    std::vector<int> klo;       // [n_tiles] first node of each tile's slab, a multiple of 4
    std::vector<unsigned> tile_ref;       // [2][n_tiles] first bin at rest (centres, lower edges) in 2^-fb nodes
    std::vector<float> lane_node, lane_rest;  // [32] lane * dt/dj at rest: whole nodes, rest
};

// entries: 8-byte entries that fit the slab's shared memory; beta: the line-of-sight
// speed the Doppler halo covers, over c; bands: a fixed number of age bands (0 = by
// cost).
inline SlabLayout slab_layout(int n_age, int n_Z, double ls0, double dls, int n_lambda, double lambda0, double dlambda,
                              double z_cosmo, long long entries, double beta, int fixed_bands) {
    // a slab per tile and age band: a band's age pairs (an odd number of entries per
    // node) over the nodes of the tile's R rounds plus the Doppler halo. Among the
    // band sizes that fit, take the one with the lowest estimated cost per particle:
    // n_tiles * (per-particle setup + R rounds + bands).
    SlabLayout L;
    const int ca = std::max(n_age - 1, 1);
    const double A0 = dlambda / ((1.0 + z_cosmo) * dls);
    const double a_lo = A0 / (1.0 + beta), a_hi = A0 / (1.0 - beta);
    const double lam_max = (lambda0 + (n_lambda - 1) * dlambda) / (1.0 + z_cosmo);
    const int shift = (int)std::ceil(lam_max / dls * beta / (1.0 - beta));
    L.nzc = std::max(n_Z, 2);
    // kind 0 covers dt/dj in (30/31, 1] (and the two-read rounds just above 1)
    // when the halo's range reaches it; kind 1 dt/dj in [1/2, 1); else kind 2
    L.kind = (a_lo > 30.0 / 31.0 && a_lo < 1.0) ? 0 : ((a_lo >= 0.5 && a_hi < 0.999) ? 1 : 2);
    const int B = kind_bins(L.kind);
    struct Geo { int apb, bands, pitch, slab_w, R, last, need; double cost; };
    Geo best{0, 0, 0, 0, 0, 0, 0, 1e300};
#define RUBIX_R(r) r,
    const int rounds[] = {RUBIX_ROUNDS(RUBIX_R)};
#undef RUBIX_R
    for (int apb = ca; apb >= 1; --apb) {
        const int bands = (ca + apb - 1) / apb;
        if (bands > kMaxBands) break;
        if (fixed_bands > 0 && bands != std::min(fixed_bands, ca)) continue;
        const int pitch = (apb * L.nzc) | 1;
        const int slab_max = (int)std::min<long long>(entries / pitch, 1 << 14) / 4 * 4;
        for (int r : rounds) {
            // bins of the last lane of the last round, deposit (also a mean
            // round more) and adjoint (rounds of 32 bins, of 31 edges for means)
            const int last = std::max({B * (r - 1) + 31, (B - 1) * r + r + 1, (B * r + 31) / 32 * 32 - 1});
            const int need = (int)std::ceil((last + 1) * std::max(a_hi, 1.0)) + 3;
            if (need + 2 * shift + 8 > slab_max) continue;
            // a slab twice the halo wide at most: more would only be staged
            const int slab_w = std::min(slab_max, (need + 4 * shift + 11) / 4 * 4);
            const int n_tiles = (n_lambda + B * r - 1) / (B * r);
            const double cost = n_tiles * (40.0 + 15.0 * r + 6.0 * bands);
            if (cost < best.cost) best = Geo{apb, bands, pitch, slab_w, r, last, need, cost};
        }
    }
    // no slab fits (very wide Doppler halo): global-memory path only (need = 0 =
    // slab_w fails every kernel's test for a fast path)
    if (best.R == 0) best = Geo{ca, 1, (ca * L.nzc) | 1, 0, 1, 0, 0, 0.0};
    L.rounds = best.R;
    L.apb = best.apb;
    L.n_bands = best.bands;
    L.pitch = best.pitch;
    L.slab_w = best.slab_w;
    L.last = best.last;
    L.need = best.need;
    // bin `last` of a particle reads up to node floor(f + last A) + 1, f < 1. (With
    // the halo's a_hi as the limit, particles that approach left the rounds at 800
    // km/s, receding ones where the slab ends: 1495 km/s on a grid of 3 A bins.)
    L.a_max = (float)std::max(a_hi, (best.need - 3.0) / std::max(best.last, 1) - 1e-6);
    L.tile_w = B * best.R;
    L.n_tiles = (n_lambda + L.tile_w - 1) / L.tile_w;
    for (int m = 0; m < 2; ++m) {
        L.ib[m] = (float)std::floor((B - m) * A0 + 0.5);
        L.fbr[m] = (float)((B - m) * A0 - L.ib[m]);
    }
    L.a0_1m = (float)(1.0 - A0);
    // fixed point of the Doppler shifts: fb bits after the point, such that a
    // position anywhere in a slab's margin fits 32 bits and the shift per bin
    // (|g| <= A0 beta / (1 - beta), times 2^(fb + 13)) 31
    L.fb = 26;
    while (L.fb > 0 && ((L.slab_w - L.need + 4.0) * std::ldexp(1.0, L.fb) >= 4294967296.0 ||
                        A0 * beta / (1.0 - beta) * std::ldexp(1.0, L.fb + 13) >= 2147483648.0))
        --L.fb;
    L.jc = n_lambda > 4096 ? 4096 : 0;
    L.klo.assign(L.n_tiles, 0);
    L.tile_ref.assign(2 * (size_t)L.n_tiles, 0u);
    L.s_min = -1e30f;
    L.s_max = 1e30f;
    for (int t = 0; t < L.n_tiles; ++t) {
        // nodes the tile's fast path reads: K0 .. K0 + need - 1 with K0 within
        // +-shift of the zero-velocity position t00 of its first bin
        const int j0 = t * L.tile_w;
        const double t00 = ((lambda0 + j0 * dlambda) / (1.0 + z_cosmo) - ls0) / dls;
        const double k = std::floor((t00 - shift - 1.0 - 0.5 * (L.slab_w - L.need - 2 * shift - 8)) / 4.0) * 4.0;
        L.klo[t] = (int)std::max(-1e6, std::min(k, 1e6));
        for (int m = 0; m < 2; ++m) {
            const double c = t00 - 0.5 * A0 * m - L.klo[t];  // at rest, from the slab's first node
            if (L.slab_w > 0 && std::abs(t00) < 9e5)
                L.tile_ref[(size_t)m * L.n_tiles + t] = (unsigned)std::llround(std::ldexp(c, L.fb));
            else
                L.s_max = -1e30f;  // no slab, or bins absurdly far from the templates: per-bin path
            // a particle's first node K0 in [0, slab_w - need) for every tile
            L.s_min = std::max(L.s_min, (float)(0.01 - c));
            L.s_max = std::min(L.s_max, (float)(L.slab_w - L.need - 0.01 - c));
        }
    }
    for (int l = 0; l < 32; ++l) {
        const double w = std::floor(l * A0);
        L.lane_node.push_back((float)w);
        L.lane_rest.push_back((float)(l * A0 - w));
    }
    return L;
}

}  // namespace rubix
