// deposit_kernel.cuh -- SSP lookup, Doppler shift, resampling and per-spaxel
// sum (Sec. 3: every star's spectrum is taken from an SSP library by age and
// metallicity, shifted by its line-of-sight velocity, resampled onto the
// instrument's wavelength grid and added to the spaxel it falls in).
//
// K3 (k_setup, setup.cu) has turned each in-field particle, in sorted order,
// into a 32-byte record (DepRec): its four mass-scaled bilinear corner weights,
// its cell's entry in the age band, its Doppler shift against a particle at rest in
// fixed point, and which rounds it takes; and into a 16-byte record (MapRec) with
// the full affine map t(j) = B + jA from output bin j to the fractional SSP node
// position, for the per-bin path and the adjoint.
//
// The templates are kept, for the deposit, as age pairs: entry (ia, iz) of a
// node holds T(ia, iz) and T(ia+1, iz), so that a cell's four corners are two
// neighbouring 8-byte entries. An age band's entries are stored contiguously,
// node-major with an odd number of entries per node. Against one 16-byte quad
// per cell the pairs cost one more load instruction per round (the same
// shared-memory wavefronts) and halve a node's bytes: bands of twice the
// ages fit the same slab, so each work item's row is visited half as often.
//
// K4 (k_deposit) is persistent: each CTA owns a contiguous, cost-balanced range
// of (wavelength tile, work item) pairs, a work item being <= chunk particles
// of one spaxel. For each tile and age band the CTA stages the band's entries
// over the tile's node range plus a Doppler halo in shared memory (bulk copies;
// 16-bit templates are widened by the CTA's threads), and its warps accumulate
// whole items in registers in a fixed particle order. Particles are sorted by
// (spaxel, age band), so for band b each item's band-b particles are
// contiguous; band 0 writes the item's row and later bands continue it.
//
// One warp takes one particle at a time, R rounds of kBins bins (kinds in
// slab_layout.h). A lane forms M = sum_c w_c T_c at its node and interpolates to the
// next node's value, which it takes from another lane by one shuffle (kinds 0
// and 1) or from its own second read. Node positions of the rounds do not
// depend on one another (tile.cuh), so that the rounds' loads can all be in
// flight. Particles that no rounds fit (Doppler shifts beyond the slab's halo)
// take a per-bin path.
//
// Spaxels with more than `chunk` particles are split into several items whose
// FP32 partial rows K5 (rows.cu) adds in item order, so the cube is bitwise
// reproducible. Each later age band continues the row the earlier bands left:
// the warp that owns the item in that band loads the row segment into its
// accumulators before its particles and stores it back after them (plain
// loads and stores, no atomics; one owner per row and band, bands separated
// by the CTA barrier, so the order of every addition is fixed).
#pragma once

#include "common.cuh"
#include "kernels.h"
#include "tile.cuh"

namespace rubix {

// ----------------------------------------------------------------------------
// Per-bin path.
// ----------------------------------------------------------------------------
// Do bins j and j + span have their nodes in the slab?
static __device__ __noinline__ bool bins_in_slab(const float4 g4, const TileCtx C, int j, int span, bool owned) {
    if (!owned || j >= C.n_lambda) return true;
    const int c0_bi = __float_as_int(g4.x);
    const int e = rec_entry(c0_bi, C);
    if ((unsigned)e >= (unsigned)max(C.pitch - 1, 0)) return false;
    float f;
    const int ka = node_pos(j, rec_bi(c0_bi), g4.y, g4.z, g4.w, f) - C.klo;
    const int kb = node_pos(j + span, rec_bi(c0_bi), g4.y, g4.z, g4.w, f) - C.klo;
    return ka >= 0 && kb + 1 < C.slab_w;
}

// Spectrum value of one particle at bin j (0 for bins the lane does not own); all
// lanes of the warp take part. From the global array a warp's loads touch a line per
// lane and node, so the next node's value is the next lane's own where that lane is
// on it (1e5 particles with a dispersion of 2000 km/s: 3890 us without, 2710 with).
static __device__ __noinline__ float bin_value(const float4 w4, const float4 g4, const TileCtx C, int j, bool owned,
                                        bool use_slab) {
    const bool in = owned && j < C.n_lambda;
    const int c0_bi = __float_as_int(g4.x);
    const int e = rec_entry(c0_bi, C);
    float f;
    const int k = node_pos(j, rec_bi(c0_bi), g4.y, g4.z, g4.w, f);
    if (use_slab) {
        if (!in) return 0.f;
        const float s0 = quad_dot(w4, quad_at(C, true, e, k)), s1 = quad_dot(w4, quad_at(C, true, e, k + 1));
        return fmaf(f, s1 - s0, s0);
    }
    const float m0 = in ? quad_dot(w4, quad_global(C, e, k)) : 0.f;
    const int lane = threadIdx.x & 31;
    const int kn = __shfl_down_sync(0xffffffffu, in ? k : INT_MIN, 1);
    float m1 = __shfl_down_sync(0xffffffffu, m0, 1);
    if (!in) return 0.f;
    if (lane == 31 || kn != k + 1) m1 = quad_dot(w4, quad_global(C, e, k + 1));
    return fmaf(f, m1 - m0, m0);
}

// Bin j's mean: M integrated segment by segment over [e_j, e_{j+1}].
static __device__ __noinline__ float mean_value(const float4 w4, const float4 g4, const TileCtx C, int j, bool owned,
                                         bool use_slab) {
    if (!owned || j >= C.n_lambda) return 0.f;
    const int c0_bi = __float_as_int(g4.x);
    const int e = rec_entry(c0_bi, C);
    float fa, fb;
    const int ka = node_pos(j, rec_bi(c0_bi), g4.y, g4.z, g4.w, fa);
    const int kb = node_pos(j + 1, rec_bi(c0_bi), g4.y, g4.z, g4.w, fb);
    auto node = [&](int k) { return quad_dot(w4, quad_at(C, use_slab, e, k)); };
    // segments [k, k + 1] outside [-1, n_ls] are zero
    const int k_first = max(ka, -1), k_last = min(kb, C.n_ls - 1);
    float s = 0.f;
    float m0 = node(k_first);
    for (int k = k_first; k <= k_last; ++k) {
        const float m1 = node(k + 1);
        const float u0 = (k == ka) ? fa : 0.f, u1 = (k == kb) ? fb : 1.f;
        s = fmaf(u1 - u0, fmaf(m1 - m0, 0.5f * (u0 + u1), m0), s);
        m0 = m1;
    }
    const float len = (float)(kb - ka) + (fb - fa);
    if (len > 0.f) return s / len;
    const float ma = node(ka);  // a bin narrower than FP32 resolves: the edge value
    return fmaf(fa, node(ka + 1) - ma, ma);
}

// Every bin on the per-bin path, from the slab if every bin of the warp has its
// nodes there, else from the global array. NR rounds of B bins; the last holds
// LAST bins.
template <int NR, int B, int LAST, bool MEAN>
__device__ __forceinline__ void general_particle(const float4 w4, const float4 g4, const TileCtx& C, int lane,
                                                 float (&acc)[NR], unsigned long long* slow_count) {
    bool ok = true;
#pragma unroll
    for (int i = 0; i < NR; ++i)
        ok = ok && bins_in_slab(g4, C, C.j0 + B * i + lane, MEAN ? 1 : 0, lane < (i < NR - 1 ? B : LAST));
    const bool use_slab = C.slab_w > 0 && __all_sync(0xffffffffu, ok);
    if (!use_slab && lane == 0 && slow_count) atomicAdd(slow_count, 1ull);
#pragma unroll
    for (int i = 0; i < NR; ++i) {
        const int j = C.j0 + B * i + lane;
        const bool owned = lane < (i < NR - 1 ? B : LAST);
        acc[i] += MEAN ? mean_value(w4, g4, C, j, owned, use_slab) : bin_value(w4, g4, C, j, owned, use_slab);
    }
}

// ----------------------------------------------------------------------------
// Rounds at bin centres.
// ----------------------------------------------------------------------------
// Kind 0, A = 1 - delta with delta in [0, 1/31): lane l of round r reads node
// K0 + 31 r + o_r + l, o_r = floor(x_r), x_r = f - 31 r delta. Its bin sits g =
// frac(x_r) - l delta in (-1, 1) from that node: the value is M + |g| (X - M)
// with X the neighbour on g's side, from lane l -+ 1.
template <int R>
__device__ __forceinline__ void rounds_near1(const float4 w4, const TileCtx& C, uint32_t base, float f, float delta,
                                             int lane, float lanef, float (&acc)[R]) {
    const uint32_t p8 = (uint32_t)C.pitch * 8u;
    base -= kMagicBits * p8;
    const float nld = __fmul_rn(-lanef, delta);
    const float fb = __fmul_rn(-31.f, delta);
#pragma unroll
    for (int r = 0; r < R; r += 2) {
        const int r1 = r + 1 < R ? r + 1 : r;
        const float2 mg = make_float2(kMagic + 31.f * r, kMagic + 31.f * r1);
        const float2 x = __ffma2_rn(make_float2((float)r, (float)r1), make_float2(fb, fb), make_float2(f, f));
        const float2 y = __fadd2_rd(x, mg);
        const float2 fl = __fadd2_rn(y, make_float2(-mg.x, -mg.y));
        const float2 g = __fadd2_rn(__fadd2_rn(x, make_float2(-fl.x, -fl.y)), make_float2(nld, nld));
        const float Ma = quad_dot(w4, lds_quad(base + __float_as_uint(y.x) * p8, C));
        // the sign of g picks the lane: (bits of g in (-2, 2)) >> 30 is -2 or 0
        const float Xa = __shfl_sync(0xffffffffu, Ma, lane + 1 + (__float_as_int(g.x) >> 30));
        if (r + 1 < R) {
            const float Mb = quad_dot(w4, lds_quad(base + __float_as_uint(y.y) * p8, C));
            const float Xb = __shfl_sync(0xffffffffu, Mb, lane + 1 + (__float_as_int(g.y) >> 30));
            const float2 D = __fadd2_rn(make_float2(Xa, Xb), make_float2(-Ma, -Mb));
            const float2 v = __ffma2_rn(make_float2(fabsf(g.x), fabsf(g.y)), D, make_float2(Ma, Mb));
            const float2 a = __fadd2_rn(make_float2(acc[r], acc[r1]), v);
            acc[r] = a.x;
            acc[r1] = a.y;
        } else {
            acc[r] += fmaf(fabsf(g.x), Xa - Ma, Ma);
        }
    }
}

// Kind 1 (A in [1/2, 1 - kShuffleTol)) and the two-read rounds (any A): lane l reads
// its bin's node n_l. In kind 1 the next node is lane l + 1's, or lane l + 2's
// when lane l + 1 has the same node (phi_l + A < 1). Near that limit (within
// the rounding of phi, kShuffleTol / 2) lane l + 2 holds node n_l + 1 in either case,
// since 1 - A > kShuffleTol.
template <int R, int B, bool SHUFFLE>
__device__ __forceinline__ void rounds_phi(const float4 w4, const TileCtx& C, const LanePos& L, float ib, float delta,
                                           int lane, float (&acc)[R]) {
    const uint32_t p8 = (uint32_t)C.pitch * 8u;
    const uint32_t sib = (uint32_t)(int)ib * p8;
    const float dt = -(delta + 0.5f * kShuffleTol);
    uint32_t base = L.base;
#pragma unroll
    for (int r = 0; r < R; r += 2) {
        const int r1 = r + 1 < R ? r + 1 : r;
        const float2 x = __ffma2_rn(make_float2((float)r, (float)r1), make_float2(L.fb, L.fb), make_float2(L.x0, L.x0));
        const float2 y = __fadd2_rd(x, make_float2(kMagic, kMagic));
        const float2 fl = __fadd2_rn(y, make_float2(-kMagic, -kMagic));
        const float2 phi = __fadd2_rn(x, make_float2(-fl.x, -fl.y));
        const uint32_t aa = base + __float_as_uint(y.x) * p8;
        base += sib;
        const float Ma = quad_dot(w4, lds_quad(aa, C));
        float Xa, Xb, Mb;
        if (SHUFFLE) {
            const float2 s = __fadd2_rn(phi, make_float2(dt, dt));
            Xa = __shfl_sync(0xffffffffu, Ma, lane + 1 - (__float_as_int(s.x) >> 31));
            if (r + 1 < R) {
                Mb = quad_dot(w4, lds_quad(base + __float_as_uint(y.y) * p8, C));
                Xb = __shfl_sync(0xffffffffu, Mb, lane + 1 - (__float_as_int(s.y) >> 31));
            }
        } else {
            Xa = quad_dot(w4, lds_quad(aa + p8, C));
            if (r + 1 < R) {
                const uint32_t ab = base + __float_as_uint(y.y) * p8;
                Mb = quad_dot(w4, lds_quad(ab, C));
                Xb = quad_dot(w4, lds_quad(ab + p8, C));
            }
        }
        if (r + 1 < R) {
            base += sib;
            const float2 D = __fadd2_rn(make_float2(Xa, Xb), make_float2(-Ma, -Mb));
            const float2 v = __ffma2_rn(phi, D, make_float2(Ma, Mb));
            const float2 a = __fadd2_rn(make_float2(acc[r], acc[r1]), v);
            acc[r] = a.x;
            acc[r1] = a.y;
        } else {
            acc[r] += fmaf(phi.x, Xa - Ma, Ma);
        }
    }
}

// A in (1, kGatherMax): a round's 32 bins lie on up to 64 nodes. Lanes on their
// own bins' nodes would collide on the banks (nodes 16 apart share one: the two
// reads per bin took 16 wavefronts, half of them conflicts), so lane l reads
// nodes n_0 + l and, as far as the round reaches, n_0 + 32 + l, conflict-free,
// and each bin takes its two nodes' M from those lanes: 7 to 8 wavefronts and
// four shuffles. Survey grid (dt/dj 1.58, 5e5 particles): 1003 -> 961 us per
// forward; the chain of a round is longer, so CTAs of few items (1e4 particles:
// 112 us, 120 with it) read twice.
constexpr float kGatherMax = 1.95f;
template <int R, int B>
__device__ __forceinline__ void rounds_gather(const float4 w4, const TileCtx& C, const LanePos& L, uint32_t base0,
                                              float f, float ib, int il, int hi, int lane, float (&acc)[R]) {
    const uint32_t p8 = (uint32_t)C.pitch * 8u;
    const uint32_t sib = (uint32_t)(int)ib * p8;
#pragma unroll
    for (int r = 0; r < R; r += 2) {
        const int r1 = r + 1 < R ? r + 1 : r;
        const float2 rr = make_float2((float)r, (float)r1), fb2 = make_float2(L.fb, L.fb);
        const float2 mg = make_float2(kMagic, kMagic);
        const float2 x = __ffma2_rn(rr, fb2, make_float2(L.x0, L.x0));
        const float2 y = __fadd2_rd(x, mg);
        const float2 fl = __fadd2_rn(y, make_float2(-kMagic, -kMagic));
        const float2 phi = __fadd2_rn(x, make_float2(-fl.x, -fl.y));
        const float2 y0 = __fadd2_rd(__ffma2_rn(rr, fb2, make_float2(f, f)), mg);  // lane 0's
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            if (r + h >= R) break;
            const int b0 = __float_as_int(h ? y0.y : y0.x);
            const uint32_t a = base0 + (uint32_t)b0 * p8;
            base0 += sib;
            const int k = il + __float_as_int(h ? y.y : y.x) - b0;  // the bin's node, from lane 0's
            const float Ma = quad_dot(w4, lds_quad(a, C));
            float Mb = 0.f;
            if (lane <= hi) Mb = quad_dot(w4, lds_quad(a + 32u * p8, C));
            const float sa = __shfl_sync(0xffffffffu, Ma, k), sb = __shfl_sync(0xffffffffu, Mb, k);
            const float ta = __shfl_sync(0xffffffffu, Ma, k + 1), tb = __shfl_sync(0xffffffffu, Mb, k + 1);
            const float m0 = k < 32 ? sa : sb, m1 = k < 31 ? ta : tb;
            acc[r + h] += fmaf(h ? phi.y : phi.x, m1 - m0, m0);
        }
    }
}

// ----------------------------------------------------------------------------
// Rounds of bin means (flux-conserving resampling). The record maps j to bin
// j's lower edge e_j = t(j) - A/2 (node units); bin j's value is the mean of
// the weighted template's linear interpolant M(t) over [e_j, e_{j+1}]. A tile
// of B R bins is R rounds of B - 1 bins and a last round of R bins; lane l of
// a round owns edge l and bin l between edges l and l + 1.
//
// Kind 0: as at bin centres, lane l reads node K0 + o_r + l and takes the
// neighbour's M on g's side, which gives the interpolant at its edge, L_l. The
// interval of bin l holds at most one node, K = K0 + o_r + l + (g >= 0), whose
// M is that neighbour's or the lane's own; with a the distance from edge l to K
// and b = A - a, the trapezoids on both sides of K give
//   mean = M_K / 2 + (a L_l + b L_{l+1}) / (2A),
// which also holds with no node inside (b < 0: the three points lie on one
// line). L_{l+1} is one more shuffle.
// ----------------------------------------------------------------------------
template <int R>
__device__ __forceinline__ void mean_rounds_near1(const float4 w4, const TileCtx& C, uint32_t base, float f,
                                                  float delta, int lane, float lanef, float (&acc)[R + 1]) {
    // with the weights halved (M' = M/2, L' = L/2), and a L + b L_{l+1} =
    // a (L - L_{l+1}) + A L_{l+1}, the mean is M'_K + L'_{l+1} + (a/A)(L' - L'_{l+1})
    const float4 wh = make_float4(0.5f * w4.x, 0.5f * w4.y, 0.5f * w4.z, 0.5f * w4.w);
    const uint32_t p8 = (uint32_t)C.pitch * 8u, s30 = 30u * p8, s29 = 29u * p8;
    const float nld = __fmul_rn(-lanef, delta);
    const float d30 = __fmul_rn(30.f, delta);
    const float iA = 1.f / (1.f - delta);
    const int lp = lane + 1, lm = lane - 1;
    // the round's first node and fraction are carried from round to round (the
    // closed form of rounds_near1 measured 5 % slower here: more registers)
#pragma unroll
    for (int r = 0; r + 1 <= R; r += 2) {
        // the last round (R bins): lanes above R + 1 read nothing
        Quad Qa = lds_quad(base, C), Qb;
        Qb.a = Qb.b = make_float2(0.f, 0.f);
        const float fa = f;
        f -= d30;
        bool carry = f < 0.f;
        f = carry ? f + 1.f : f;
        base += carry ? s29 : s30;
        if (r + 1 < R || lane <= R + 1) Qb = lds_quad(base, C);
        const float fb = f;
        if (r + 2 <= R) {
            f -= d30;
            carry = f < 0.f;
            f = carry ? f + 1.f : f;
            base += carry ? s29 : s30;
        }
        const float2 M = make_float2(quad_dot(wh, Qa), quad_dot(wh, Qb));
        const float2 g = __fadd2_rn(make_float2(fa, fb), make_float2(nld, nld));
        const bool ua = g.x >= 0.f, ub = g.y >= 0.f;
        const float2 X = make_float2(__shfl_sync(0xffffffffu, M.x, ua ? lp : lm),
                                     __shfl_sync(0xffffffffu, M.y, ub ? lp : lm));
        const float2 Lv = __ffma2_rn(make_float2(fabsf(g.x), fabsf(g.y)), __fadd2_rn(X, make_float2(-M.x, -M.y)), M);
        const float2 Ln = make_float2(__shfl_down_sync(0xffffffffu, Lv.x, 1), __shfl_down_sync(0xffffffffu, Lv.y, 1));
        const float2 MK = make_float2(ua ? X.x : M.x, ub ? X.y : M.y);
        const float2 ai = __ffma2_rn(make_float2(-g.x, -g.y), make_float2(iA, iA),
                                     make_float2(ua ? iA : 0.f, ub ? iA : 0.f));
        const float2 v = __ffma2_rn(ai, __fadd2_rn(Lv, make_float2(-Ln.x, -Ln.y)), __fadd2_rn(MK, Ln));
        const float2 a = __fadd2_rn(make_float2(acc[r], acc[r + 1]), v);
        acc[r] = a.x;
        acc[r + 1] = a.y;
    }
    if (!(R & 1)) {
        // R + 1 rounds, odd: the last round (R bins) alone
        Quad Q;
        Q.a = Q.b = make_float2(0.f, 0.f);
        if (lane <= R + 1) Q = lds_quad(base, C);
        const float M = quad_dot(wh, Q);
        const float g = __fadd_rn(f, nld);
        const bool up = g >= 0.f;
        const float X = __shfl_sync(0xffffffffu, M, up ? lp : lm);
        const float L = fmaf(fabsf(g), X - M, M);
        const float Ln = __shfl_down_sync(0xffffffffu, L, 1);
        const float ai = fmaf(-g, iA, up ? iA : 0.f);
        acc[R] += fmaf(ai, L - Ln, (up ? X : M) + Ln);
    }
}

// Any A in [1/2, 2): lane l reads both nodes of its edge, n_l and n_l + 1, and
// takes L, M(n) and n of edge l + 1 from lane l + 1. With d = n_{l+1} - n_l in
// {0, 1, 2}, the trapezoids from edge l to node n_l + 1, from there to n_{l+1}
// (a length of d - 1 segments: none, one, or minus the whole segment that
// holds both edges) and on to edge l + 1 give
//   2 A mean = (1 - phi_l)(L_l + M(n_l + 1)) + (d - 1)(M(n_l + 1) + M(n_{l+1}))
//              + phi_{l+1} (M(n_{l+1}) + L_{l+1}).
template <int R, int B>
__device__ __forceinline__ void mean_rounds_phi(const float4 w4, const TileCtx& C, const LanePos& L, float ib, float A,
                                                int lane, float (&acc)[R + 1]) {
    const float iA = 0.5f / A;
    const uint32_t p8 = (uint32_t)C.pitch * 8u;
    const uint32_t sib = (uint32_t)(int)ib * p8;
    uint32_t base = L.base;
#pragma unroll
    for (int r = 0; r <= R; ++r) {
        const float x = fmaf((float)r, L.fb, L.x0);
        const float y = __fadd_rd(x, kMagic);
        const float fl = y - kMagic;
        const float phi = x - fl;
        float M0 = 0.f, M1 = 0.f;
        if (r < R || lane <= R) {  // the last round has R bins, R + 1 edges
            const uint32_t a = base + __float_as_uint(y) * p8;
            M0 = quad_dot(w4, lds_quad(a, C));
            M1 = quad_dot(w4, lds_quad(a + p8, C));
        }
        base += sib;
        const float Lv = fmaf(phi, M1 - M0, M0);
        const float n = L.nf + fl;
        const float Ln = __shfl_down_sync(0xffffffffu, Lv, 1);
        const float Mn = __shfl_down_sync(0xffffffffu, M0, 1);
        const float d = __shfl_down_sync(0xffffffffu, n, 1) - n;
        const float ph1 = (phi + A) - d;  // phi of edge l + 1
        const float v = fmaf(1.f - phi, Lv + M1, fmaf(d - 1.f, M1 + Mn, ph1 * (Mn + Ln)));
        acc[r] = fmaf(iA, v, acc[r]);
    }
}

// What the rounds of a (tile, job) share: the tile's first bin at rest in the
// records' fixed point (SlabParams::tile_ref), and the lane's constants.
struct RoundCtx {
    int jrel;            // (j0 - jc) << 19: times DepRec::g, high word = the shift since jc
    uint32_t ref;
    int fb;
    float fscale;        // 2^-fb
    float a0_1m;
    float ib, fbr;       // whole nodes of a round and the rest, at rest
    float il, fl;        // whole nodes of the lane's bins and the rest, at rest
    bool gather;         // enough work in the CTA for rounds_gather
};

// Adds one particle's spectrum to acc (setup by every lane; warp-uniform path).
template <int R, int KIND, bool MEAN, int NR>
__device__ __forceinline__ void deposit_particle(const float4 w4, const float4 r4, const float4* __restrict__ map4,
                                                 const TileCtx& C, const RoundCtx& T, int lane, float lanef,
                                                 float (&acc)[NR], unsigned long long* slow_count) {
    constexpr int B = kind_bins(KIND), BR = MEAN ? B - 1 : B;
    const unsigned ef = __float_as_uint(r4.w);
    const uint32_t p = (uint32_t)(__mulhi(T.jrel, __float_as_int(r4.y)) + __float_as_int(r4.x)) + T.ref;
    const uint32_t p8 = (uint32_t)C.pitch * 8u;
    const uint32_t kw = p >> T.fb;  // first node, from the slab's
    const float f = (float)(p & ((1u << T.fb) - 1u)) * T.fscale;
    if ((ef >> 30) == kPathMain && KIND == 0) {
        const uint32_t base = C.slab + (kw + (uint32_t)lane) * p8 + ef;
        if constexpr (MEAN) mean_rounds_near1<R>(w4, C, base, f, r4.z, lane, lanef, acc);
        else rounds_near1<R>(w4, C, base, f, r4.z, lane, lanef, acc);
    } else if ((ef >> 30) != kPathBins) {
        const float da = KIND == 0 ? T.a0_1m - r4.z : r4.z;  // dt/dj less that at rest
        LanePos L;
        L.x0 = fmaf(lanef, da, f + T.fl);
        L.fb = fmaf((float)BR, da, T.fbr);
        L.base = C.slab + (kw + (uint32_t)(int)T.il) * p8 + (ef & 0x3fffffffu) - kMagicBits * p8;
        const float delta = T.a0_1m - da;
        if constexpr (MEAN) {
            L.nf = (float)kw + T.il;
            mean_rounds_phi<R, B>(w4, C, L, T.ib, 1.f - delta, lane, acc);
        } else {
            if (KIND == 1 && (ef >> 30) == kPathMain) rounds_phi<R, B, true>(w4, C, L, T.ib, delta, lane, acc);
            else if (KIND == 2 && T.gather && delta < -0.03f && delta > 1.f - kGatherMax) {
                // lanes of the second read: up to node floor(31 dt/dj) + 2 of the round's
                const uint32_t base0 = C.slab + (kw + (uint32_t)lane) * p8 + (ef & 0x3fffffffu) - kMagicBits * p8;
                rounds_gather<R, B>(w4, C, L, base0, f, T.ib, (int)T.il, (int)(31.f * (1.f - delta)) + 2 - 32, lane, acc);
            } else rounds_phi<R, B, false>(w4, C, L, T.ib, delta, lane, acc);
        }
    } else {
        const float4 g4 = *map4;
        if (g4.z > 0.f)  // a_hi = 0 marks a spectrum that misses every bin
            general_particle<NR, BR, MEAN ? R : B, MEAN>(w4, g4, C, lane, acc, slow_count);
    }
}

constexpr int kJobChunk = 32;  // jobs per shared-memory work table

// One work item's particles [q0, q1) of the current band, accumulated in
// registers in sorted order onto the item's row dst (zero for band 0, the
// earlier bands' sum for later bands), then stored.
template <int R, int KIND, bool MEAN>
__device__ __forceinline__ void deposit_item(const DepositParams& P, const TileCtx& C, const DepJob& J, int t, int q0,
                                             int q1, float* dst, int band, int lane, float lanef, float2 lref, bool gather) {
    constexpr int B = kind_bins(KIND), BR = MEAN ? B - 1 : B, NR = MEAN ? R + 1 : R;
    const float4* __restrict__ rec4 = reinterpret_cast<const float4*>(J.rec);
    // the next particle's record is pulled into L1 while the current one is
    // deposited (no registers held across the particle)
    if (q0 < q1) asm volatile("prefetch.global.L1 [%0];" ::"l"(rec4 + 2 * q0));
    float acc[NR];
    // band 0 starts the row from zero; later bands continue the row the
    // earlier bands left (loaded now, in flight while the first particle's
    // record and setup are prepared), so the row is written back with plain
    // stores and no atomics
    const bool full = C.j0 + B * R <= P.n_lambda;
    dst += C.j0 + lane;
    const int left = full ? 1 << 20 : P.n_lambda - C.j0 - lane;  // bins from the lane's first to the row's end
#pragma unroll
    for (int r = 0; r < NR; ++r) {
        const bool owned = lane < (MEAN && r == R ? R : BR);
        acc[r] = (band > 0 && owned && BR * r < left) ? dst[BR * r] : 0.f;
    }
    RoundCtx T;
    T.jrel = (int)((unsigned)(C.j0 - P.jc) << 19);
    T.ref = P.tile_ref[(MEAN ? P.n_tiles : 0) + t];
    T.fb = P.fb;
    T.fscale = __int_as_float((127 - P.fb) << 23);
    T.a0_1m = P.a0_1m;
    T.ib = P.ib[MEAN];
    T.fbr = P.fbr[MEAN];
    T.il = lref.x;
    T.fl = lref.y;
    T.gather = gather;
    for (int q = q0; q < q1; ++q) {
        if (q + 1 < q1) asm volatile("prefetch.global.L1 [%0];" ::"l"(rec4 + 2 * (q + 1)));
        const float4 w4 = rec4[2 * q], r4 = rec4[2 * q + 1];
        deposit_particle<R, KIND, MEAN, NR>(w4, r4, reinterpret_cast<const float4*>(J.map) + q, C, T, lane, lanef, acc,
                                            P.slow_count);
    }
#pragma unroll
    for (int r = 0; r < NR; ++r) {
        const bool owned = lane < (MEAN && r == R ? R : BR);
        if (owned && BR * r < left) dst[BR * r] = acc[r];
    }
}

// ----------------------------------------------------------------------------
// K4: deposit. Shared memory: kDepHeader bytes (mbarrier, counters, job work
// table), then the slab: slab_w nodes x pitch entries, node-major (entry e at
// node k at (k - klo) * pitch + e - e0). pitch is odd, so the 8-byte entries
// that 16 lanes read at consecutive nodes fall in distinct bank pairs.
// ----------------------------------------------------------------------------
template <int R, int KIND, bool MEANS>
__global__ void __launch_bounds__(RUBIX_DEP_THREADS, 1) k_deposit(const __grid_constant__ DepositParams P) {
    extern __shared__ __align__(1024) unsigned char smem[];
    uint64_t* bar = reinterpret_cast<uint64_t*>(smem);
    int* s_next = reinterpret_cast<int*>(smem + 16);
    int* s_nv = reinterpret_cast<int*>(smem + 20);         // work items in the current table
    int* s_job = reinterpret_cast<int*>(smem + 64);        // [kJobChunk] job of table row k
    int* s_ia = s_job + kJobChunk;                         // [kJobChunk] its first item
    int* s_pre = s_ia + kJobChunk;                         // [kJobChunk + 1] prefix of item counts
    // [kMaxJobs + 1] exclusive prefix of the jobs' per-tile costs
    long long* jc = reinterpret_cast<long long*>(smem + 64 + 4 * (3 * kJobChunk + 2));
    static_assert(64 + 4 * (3 * kJobChunk + 2) + 8 * (kMaxJobs + 1) <= kDepHeader, "header");
    static_assert(kMaxJobs <= 64, "two jobs per lane");

    const int lane = threadIdx.x & 31;
    const float lanef = (float)lane;
    const int nb = P.n_bands;
    const long long C0 = P.cost_c0;
    // per-tile cost of each job (in-field particles + cost_c0 per work item),
    // from the device-side counts, lane l taking jobs 2l and 2l + 1
    if (threadIdx.x < 32) {
        long long c[2] = {0, 0};
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int j = 2 * lane + h;
            if (j < P.n_jobs) {
                const DepJob& J = P.jobs[j];
                c[h] = J.seg_off[(long long)J.n_s * nb] + C0 * J.item_off[J.n_s];
            }
        }
        long long x = c[0] + c[1];
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const long long y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
        }
        if (2 * lane <= P.n_jobs) jc[2 * lane] = x - c[0] - c[1];
        if (2 * lane + 1 <= P.n_jobs) jc[2 * lane + 1] = x - c[1];
        if (lane == 31 && P.n_jobs == kMaxJobs) jc[kMaxJobs] = x;
    }
    __syncthreads();
    const long long CT = jc[P.n_jobs];
    if (CT <= 0) return;
    const long long total = CT * P.n_tiles;
    const long long lo = total * blockIdx.x / gridDim.x;
    const long long hi = total * (blockIdx.x + 1) / gridDim.x;
    if (lo >= hi) return;

    if (threadIdx.x == 0) {
        mbar_init(bar, 1);
        fence_mbar_init();
    }
    __syncthreads();

    TileCtx C;
    C.slab_w = P.slab_w;
    C.pitch = P.pitch;
    C.es = P.es;
    C.n_lambda = P.n_lambda;
    C.n_ls = P.n_ls;
    C.pad = P.pad;
    C.qdt = P.qdt;
    C.a_max = P.a_max;
    C.need = P.need;
    C.slab = smem_addr(smem + kDepHeader);
#if RUBIX_DEBUG
    C.err = P.err;
#endif
    uint32_t phase = 0;
    const float2 lref = P.lane_ref[lane];

    for (long long t = lo / CT; t < P.n_tiles && t * CT < hi; ++t) {
        const long long a = max(lo - t * CT, 0ll), b = min(hi - t * CT, CT);
        if (a >= b) continue;
        // jobs overlapping the CTA's cost range [a, b) of this tile
        const int ja = upper_bound_ll(jc, P.n_jobs + 1, a) - 1;
        const int jb = min(upper_bound_ll(jc, P.n_jobs + 1, b - 1), P.n_jobs);
        C.klo = P.tile_klo[t];
        C.j0 = (int)t * P.tile_w;

      for (int cj = ja; cj < jb; cj += kJobChunk) {
        __syncthreads();  // every warp is done with the previous table
        if (threadIdx.x == 0) {
            int nv = 0, k = 0;
            s_pre[0] = 0;
            for (int j = cj; j < min(jb, cj + kJobChunk); ++j, ++k) {
                const DepJob& J = P.jobs[j];
                const long long ctj = jc[j + 1] - jc[j];
                const long long aj = max(a - jc[j], 0ll), bj = min(b - jc[j], ctj);
                const long long n_items = J.item_off[J.n_s];
                const int ia = (int)item_lower_bound(J.items, n_items, C0, aj);
                const int ib = (int)item_lower_bound(J.items, n_items, C0, bj);
                s_job[k] = j;
                s_ia[k] = ia;
                nv += max(ib - ia, 0);
                s_pre[k + 1] = nv;
            }
            for (; k < kJobChunk; ++k) s_pre[k + 1] = nv;
            *s_nv = nv;
        }

        for (int band = 0; band < nb; ++band) {
            C.e0 = P.band_e0[band];
            C.gband = band_ptr(P.pair, P.qdt, P.band_stride, band);
            __syncthreads();  // all warps are done with the previous slab and rows
            if (threadIdx.x == 0) {
                *s_next = 0;
                if (C.slab_w > 0 && !C.qdt) load_slab(C, bar);
            }
            bool ok = true;
            if (C.slab_w > 0 && !C.qdt) {
                ok = mbar_wait_bounded(bar, phase, 4000000000ll);
                phase ^= 1u;
            } else if (C.slab_w > 0) {
                // 16-bit templates: every thread converts part of the slab
                fill_slab16(C);
            }
            if (__syncthreads_or(!ok)) {
                if (threadIdx.x == 0) atomicOr(P.err, kErrTmaTimeout);
                return;
            }

            const int nv = *s_nv;
            const bool many = nv >= 2 * (int)(blockDim.x >> 5);
            int v0 = 0;
            while (true) {
                const int G = claim_size(nv - v0, RUBIX_DEP_GRAB);
                if (lane == 0) v0 = atomicAdd(s_next, G);
                v0 = __shfl_sync(0xffffffffu, v0, 0);
                if (v0 >= nv) break;
                // lanes < G look up one work item each and its band segment
                int kk = 0, qb = 0, qe = 0, sp = 0, prow = -1;
                bool live = false;
                const int v = v0 + lane;
                if (lane < G && v < nv) {
                    while (s_pre[kk + 1] <= v) ++kk;  // table row holding work item v
                    const DepJob& J = P.jobs[s_job[kk]];
                    const Item I = J.items[s_ia[kk] + (v - s_pre[kk])];
                    sp = I.spaxel;
                    prow = I.part_row;
                    qb = I.begin;
                    qe = I.end;
                    if (prow >= J.part_cap || sp < 0 || sp >= J.n_s) {
                        atomicOr(P.err, kErrBadItem);
                    } else {
                        qb = max(qb, J.seg_off[(long long)sp * nb + band]);
                        qe = min(qe, J.seg_off[(long long)sp * nb + band + 1]);
                        // band 0 visits every item: it writes the row, zeros included
                        live = band == 0 || qb < qe;
                        // the item's first record, on its way to L1 before the warp reaches it
                        if (qb < qe)
                            asm volatile("prefetch.global.L1 [%0];" ::"l"(reinterpret_cast<const float4*>(J.rec) + 2 * qb));
                    }
                }
                unsigned m = __ballot_sync(0xffffffffu, live);
                while (m) {
                    const int src = __ffs(m) - 1;
                    m &= m - 1;
                    const int k = __shfl_sync(0xffffffffu, kk, src);
                    const int q0 = __shfl_sync(0xffffffffu, qb, src);
                    const int q1 = __shfl_sync(0xffffffffu, qe, src);
                    const int s = __shfl_sync(0xffffffffu, sp, src);
                    const int pr = __shfl_sync(0xffffffffu, prow, src);
                    const DepJob& J = P.jobs[s_job[k]];
                    float* dst = (pr < 0) ? J.cube + (long long)s * J.pitch
                                          : J.partials + (long long)pr * P.n_lambda;
                    if (MEANS && J.resample)
                        deposit_item<R, KIND, true>(P, C, J, (int)t, q0, q1, dst, band, lane, lanef, lref, many);
                    else
                        deposit_item<R, KIND, false>(P, C, J, (int)t, q0, q1, dst, band, lane, lanef, lref, many);
                }
            }
        }
      }
    }
}

// The kernel of a kind for R rounds per tile (one translation unit per kind);
// nullptr for an R that is not built (RUBIX_ROUNDS in slab_layout.h).
typedef void (*DepositFn)(const DepositParams);
template <int KIND>
DepositFn deposit_fn(int R, bool means) {
    switch (R) {
#define RUBIX_DEP_R(r) \
    case r: return means ? k_deposit<r, KIND, true> : k_deposit<r, KIND, false>;
        RUBIX_ROUNDS(RUBIX_DEP_R)
#undef RUBIX_DEP_R
        default: return nullptr;
    }
}
DepositFn deposit_fn_k0(int R, bool means);
DepositFn deposit_fn_k1(int R, bool means);
DepositFn deposit_fn_k2(int R, bool means);

}  // namespace rubix
