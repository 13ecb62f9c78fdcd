// adjoint_kernel.cuh -- the adjoint of the deposit (gradients through the
// pipeline, Abstract and Sec. 1) over the deposit's own decomposition.
//
// For particle p with unit-mass bilinear weights W_c(ta, tz), the spectrum at
// bin j is S_j = sum_c W_c lerp(T_c, t_j) and the loss sees it through
// G_j = dL/dcube0[s_p, j]. The gradient needs, per particle,
//   sm  = sum_j G_j S_j                      (dL/dm = flux_scale * sm)
//   sla = sum_j G_j dS_j/dta                 (chain rule to age outside)
//   slz = sum_j G_j dS_j/dtz                 (to Z outside)
//   sv  = sum_j G_j dS_j/dt * (t_j + ls0/dls) (times dt/dv / t_abs outside)
// All three forms are linear in the templates of the particle's cell, so the
// lanes accumulate per template entry (G_j times the interpolated entry, and
// G_j times its slope times the bin position) and apply ta and tz once per
// particle and tile. The deposit's (tile, work item, age band) partition and
// slabs carry over unchanged. Bin centres: rounds of 32 bins, lane l reading
// both nodes of its bin (any dt/dj; conflict-free up to dt/dj = 1, where the
// lanes of a half-warp read at most 16 consecutive nodes). A warp reduction per
// (particle, tile) gives part[tile][particle]; K8 adds the tiles in tile order
// with a compensated FP32 sum.
#pragma once

#include "common.cuh"
#include "kernels.h"
#include "tile.cuh"

namespace rubix {

// ---------------------------------------------------------------------------
// Per (particle, tile) sums.
// ---------------------------------------------------------------------------
struct AdjSums {
    float sm, sa, sz, sv;
};

// A node's entries, by kind. Kind 0: the deposit's age pairs, the cell's four
// corners (T00, T10), (T01, T11), and sums per corner: four corners' rounding
// errors average in each form. Kinds 1, 2: each template and its difference to
// the next age's, (T0, A0), (T1, A1), and the second entry's difference to the
// first taken at the node (lds_diff): the sums of a derivative do not cancel
// (metallicity gradient to 1e-7 where corner sums give 1e-6; the two packed
// additions per node it takes cost 6 % on kind 0's shorter rounds).
//   S = (1 - tz)(T0 + ta A0) + tz (T1 + ta A1),  dS/dta = (1 - tz) A0 + tz A1,
//   dS/dtz = (T1 - T0) + ta (A1 - A0),  A = T(next age) - T.
struct Forms {
    float m, a, z;
};
template <int KIND>
__device__ __forceinline__ Forms node_forms(const float2 w, const Quad& q) {
    const float ty = 1.f - w.y, tx = 1.f - w.x;
    Forms F;
    if (KIND == 0) {
        F.m = fmaf(ty, fmaf(w.x, q.a.y, __fmul_rn(tx, q.a.x)), __fmul_rn(w.y, fmaf(w.x, q.b.y, __fmul_rn(tx, q.b.x))));
        F.a = fmaf(ty, q.a.y - q.a.x, __fmul_rn(w.y, q.b.y - q.b.x));
        F.z = fmaf(tx, q.b.x - q.a.x, __fmul_rn(w.x, q.b.y - q.a.y));
    } else {
        F.m = fmaf(ty, fmaf(w.x, q.a.y, q.a.x), __fmul_rn(w.y, fmaf(w.x, q.b.y, q.b.x)));
        F.a = fmaf(ty, q.a.y, __fmul_rn(w.y, q.b.y));
        F.z = fmaf(w.x, q.b.y - q.a.y, q.b.x - q.a.x);
    }
    return F;
}

// The four sums from the sums over corners (kind 0) or over entries and their
// differences; U is to be scaled by su.
template <int KIND>
__device__ __forceinline__ AdjSums entry_sums(const float2 w, float su, float2 U0, float2 U1, float2 V0, float2 V1) {
    AdjSums S;
    if (KIND == 0) {
        const float tx = 1.f - w.x, ty = 1.f - w.y;
        const float w0 = tx * ty, w1 = w.x * ty, w2 = tx * w.y, w3 = w.x * w.y;
        S.sm = su * fmaf(w0, U0.x, fmaf(w1, U0.y, fmaf(w2, U1.x, __fmul_rn(w3, U1.y))));
        S.sa = su * fmaf(ty, U0.y - U0.x, __fmul_rn(w.y, U1.y - U1.x));
        S.sz = su * fmaf(tx, U1.x - U0.x, __fmul_rn(w.x, U1.y - U0.y));
        S.sv = fmaf(w0, V0.x, fmaf(w1, V0.y, fmaf(w2, V1.x, __fmul_rn(w3, V1.y))));
    } else {
        S.sm = su * (fmaf(w.x, U0.y, U0.x) + __fmul_rn(w.y, fmaf(w.x, U1.y, U1.x)));
        S.sa = su * fmaf(w.y, U1.y, U0.y);
        S.sz = su * fmaf(w.x, U1.y, U1.x);
        S.sv = fmaf(w.x, V0.y, V0.x) + __fmul_rn(w.y, fmaf(w.x, V1.y, V1.x));
    }
    return S;
}

// A node's entries as (first, second - first).
__device__ __forceinline__ Quad lds_diff(uint32_t addr, const TileCtx& C) {
    Quad q = lds_quad(addr, C);
    q.b = __fadd2_rn(q.b, make_float2(-q.a.x, -q.a.y));
    return q;
}

// General path: the tile's bins one at a time (bin j0 + 32 r + l on lane l),
// nodes from the slab when every bin of the warp has its node pair there, else
// from global memory. It reads dL/dcube0 from the spaxel's row (grow) itself,
// so that the fast path's register copy never has to be kept for this call.
template <int TW, int KIND>
static __device__ __noinline__ AdjSums adj_general(const float2 w, const float4 g4, const TileCtx C, int lane,
                                            const float* __restrict__ grow, float ls0_over) {
    const int c0_bi = __float_as_int(g4.x);
    const int e = rec_entry(c0_bi, C), bi = rec_bi(c0_bi);
    bool ok = C.slab_w > 0 && (unsigned)e < (unsigned)(C.pitch - 1);
    for (int o = lane; o < TW; o += 32) {
        const int j = C.j0 + o;
        if (j < C.n_lambda) {
            float f;
            const int k = node_pos(j, bi, g4.y, g4.z, g4.w, f) - C.klo;
            ok = ok && k >= 0 && k + 1 < C.slab_w;
        }
    }
    const bool use_slab = __all_sync(0xffffffffu, ok);
    AdjSums S{0.f, 0.f, 0.f, 0.f};
    for (int o0 = 0; o0 < TW && C.j0 + o0 < C.n_lambda; o0 += 32) {
        const int j = C.j0 + o0 + lane;
        const bool in = o0 + lane < TW && j < C.n_lambda;
        float f;
        const int k = node_pos(j, bi, g4.y, g4.z, g4.w, f);
        Forms p{0.f, 0.f, 0.f};
        if (in) p = node_forms<KIND>(w, quad_at(C, use_slab, e, k));
        // the next node's forms are the next lane's own where that lane is on it
        // (as in the deposit's per-bin path)
        const int kn = __shfl_down_sync(0xffffffffu, in ? k : INT_MIN, 1);
        Forms q{__shfl_down_sync(0xffffffffu, p.m, 1), __shfl_down_sync(0xffffffffu, p.a, 1),
                __shfl_down_sync(0xffffffffu, p.z, 1)};
        if (!in) continue;
        if (lane == 31 || kn != k + 1) q = node_forms<KIND>(w, quad_at(C, use_slab, e, k + 1));
        const float Gj = grow[j];
        S.sm = fmaf(Gj, fmaf(f, q.m - p.m, p.m), S.sm);
        S.sa = fmaf(Gj, fmaf(f, q.a - p.a, p.a), S.sa);
        S.sz = fmaf(Gj, fmaf(f, q.z - p.z, p.z), S.sz);
        S.sv = fmaf(Gj * (q.m - p.m), ((float)k + f) + ls0_over, S.sv);
    }
    return S;
}

// Kind 0 (A = dt/dj in (30/31, 1]): rounds of 31 bins. Lane l reads node K0 +
// o_r + l and the neighbouring node on its bin's side, K0 + o_r + l -+ 1; the
// round's first node and fraction are carried from round to round. The three
// forms are linear in the cell's entries, so the rounds accumulate per entry c,
// in packed FP32x2 pairs: U_c = sum_j G_j V_c(j), V_c(j) the entry
// interpolated at bin j, and T_c = sum_j G_j u_j (E_c[hi] - E_c[lo]), the slope
// between the bracketing nodes times the bin's absolute position
// u_j = t_j + ls0/dls.
template <int R>
__device__ __forceinline__ AdjSums adj_near1(const float2 w, const TileCtx& C, uint32_t base, float t0, float f,
                                             float delta, int lane, float lanef, const float (&G)[R]) {
    const uint32_t p8 = (uint32_t)C.pitch * 8u, s31 = 31u * p8, s30 = 30u * p8;
    const float nld = -lanef * delta;
    const float d31 = 31.f * delta;
    const float A = 1.f - delta;
    float u = fmaf(lanef, A, t0);  // absolute position of bin j0 + 31 r + l
    const float du = 31.f * A;
    float2 U01 = make_float2(0.f, 0.f), U23 = U01, T01 = U01, T23 = U01;
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const Quad Q = lds_quad(base, C);
        const float g = f + nld;
        // lane 31 owns no bin (G = 0); it takes node - 1, so that every read
        // stays within nodes K0 .. K0 + 31 R of the slab
        const bool neg = g < 0.f || lane == 31;
        const Quad X = lds_quad(neg ? base - p8 : base + p8, C);
        const float2 D01 = __fadd2_rn(X.a, make_float2(-Q.a.x, -Q.a.y));
        const float2 D23 = __fadd2_rn(X.b, make_float2(-Q.b.x, -Q.b.y));
        const float ag = fabsf(g);
        const float2 ag2 = make_float2(ag, ag);
        const float Gj = G[r];  // 0 for lane 31 and bins past the end
        const float2 G2 = make_float2(Gj, Gj);
        U01 = __ffma2_rn(G2, __ffma2_rn(ag2, D01, Q.a), U01);
        U23 = __ffma2_rn(G2, __ffma2_rn(ag2, D23, Q.b), U23);
        const float gu = (neg ? -Gj : Gj) * u;  // D points from this node to the neighbour
        const float2 gu2 = make_float2(gu, gu);
        T01 = __ffma2_rn(gu2, D01, T01);
        T23 = __ffma2_rn(gu2, D23, T23);
        f -= d31;
        const bool carry = f < 0.f;
        f = carry ? f + 1.f : f;
        base += carry ? s30 : s31;
        u += du;
    }
    return entry_sums<0>(w, 1.f, U01, U23, T01, T23);
}

// Any A: rounds of 32 bins, the sums as in adj_near1; lane l reads both nodes
// of its bin. The slope jumps at every node, so the node is decided with all
// the record's precision, as node_pos decides it (the same operations in
// packed form; the integer parts stay in the magic sums' low bits).
template <int TW, int NR>
__device__ __forceinline__ AdjSums adj_rounds(const float2 w, const float4 g4, const TileCtx& C, int e, int bi, float A,
                                              float u0, float lanef, const float (&G)[NR]) {
    const uint32_t p8 = (uint32_t)C.pitch * 8u;
    const uint32_t base = C.slab + ((uint32_t)(bi - C.klo) * (uint32_t)C.pitch + (uint32_t)e) * 8u - kMagicBits * p8;
    const float jl = (float)C.j0 + lanef;
    const float2 bf2 = make_float2(g4.y, g4.y), ah2 = make_float2(g4.z, g4.z), al2 = make_float2(g4.w, g4.w);
    float2 U01 = make_float2(0.f, 0.f), U23 = U01, T01 = U01, T23 = U01;
#pragma unroll
    for (int r = 0; r < NR; r += 2) {
        const int r1 = r + 1 < NR ? r + 1 : r;
        const float2 j2 = __fadd2_rn(make_float2(jl, jl), make_float2(32.f * r, 32.f * r1));
        const float2 pp = __fmul2_rn(j2, ah2);  // exact
        const float2 y1 = __fadd2_rd(pp, make_float2(kMagic, kMagic));
        const float2 pi = __fadd2_rn(y1, make_float2(-kMagic, -kMagic));
        const float2 s2 = __fadd2_rn(__fadd2_rn(pp, make_float2(-pi.x, -pi.y)), __ffma2_rn(j2, al2, bf2));
        const float2 y = __fadd2_rd(s2, y1);
        const float2 fl = __fadd2_rn(y, make_float2(-y1.x, -y1.y));
        const float2 phi = __fadd2_rn(s2, make_float2(-fl.x, -fl.y));
        const float2 u = __ffma2_rn(j2, make_float2(A, A), make_float2(u0, u0));
        const float2 gu = __fmul2_rn(make_float2(G[r], G[r1]), u);  // G is 0 for bins past the end
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            if (r + h >= NR) break;
            const uint32_t a = base + __float_as_uint(h ? y.y : y.x) * p8;
            const Quad Q = lds_diff(a, C), X = lds_diff(a + p8, C);
            const float2 D01 = __fadd2_rn(X.a, make_float2(-Q.a.x, -Q.a.y));
            const float2 D23 = __fadd2_rn(X.b, make_float2(-Q.b.x, -Q.b.y));
            const float ph = h ? phi.y : phi.x, g = G[r + h], t = h ? gu.y : gu.x;
            const float2 ph2 = make_float2(ph, ph), g2 = make_float2(g, g), t2 = make_float2(t, t);
            U01 = __ffma2_rn(g2, __ffma2_rn(ph2, D01, Q.a), U01);
            U23 = __ffma2_rn(g2, __ffma2_rn(ph2, D23, Q.b), U23);
            T01 = __ffma2_rn(t2, D01, T01);
            T23 = __ffma2_rn(t2, D23, T23);
        }
    }
    return entry_sums<1>(w, 1.f, U01, U23, T01, T23);
}

// ---------------------------------------------------------------------------
// Bin means (resample = 1). With S_j the mean of the weighted interpolant over
// [e_j, e_{j+1}] (node units, width A) and the edges moving with v as
// t' = -(t + ls0/dls) / (c (1 + v/c)), differentiating the bounds gives
//   dS_j/dv = -1/(c (1 + v/c)) [ (L_{j+1} u_{j+1} - L_j u_j) / A - S_j ]
//           = -1/(c (1 + v/c)) [ u_j (L_{j+1} - L_j) / A + L_{j+1} - S_j ],
// L_j the interpolant at edge j and u_j = e_j + ls0/dls (u_{j+1} = u_j + A);
// sv sums G_j times the bracket, and sm, sa, sz sum G_j times the bin means
// of the three weighted interpolants (M, and the a- and b-weighted forms).
// ---------------------------------------------------------------------------
template <int KIND>
static __device__ __noinline__ AdjSums adj_mean_bin(const float2 w, const float4 g4, const TileCtx C, int j, float Gj,
                                                    bool use_slab, float ls0_over) {
    AdjSums S{0.f, 0.f, 0.f, 0.f};
    const int c0_bi = __float_as_int(g4.x);
    const int e = rec_entry(c0_bi, C), bi = rec_bi(c0_bi);
    float fa, fb;
    const int ka = node_pos(j, bi, g4.y, g4.z, g4.w, fa);
    const int kb = node_pos(j + 1, bi, g4.y, g4.z, g4.w, fb);
    auto node = [&](int k) { return node_forms<KIND>(w, quad_at(C, use_slab, e, k)); };
    const float len = (float)(kb - ka) + (fb - fa);
    if (!(len > 0.f)) return S;
    const int k_first = max(ka, -1), k_last = min(kb, C.n_ls - 1);
    float im = 0.f, ia = 0.f, ib = 0.f;
    Forms p = node(k_first);
    for (int k = k_first; k <= k_last; ++k) {
        const Forms q = node(k + 1);
        const float u0 = (k == ka) ? fa : 0.f, u1 = (k == kb) ? fb : 1.f;
        const float d = u1 - u0, mid = 0.5f * (u0 + u1);
        im = fmaf(d, fmaf(q.m - p.m, mid, p.m), im);
        ia = fmaf(d, fmaf(q.a - p.a, mid, p.a), ia);
        ib = fmaf(d, fmaf(q.z - p.z, mid, p.z), ib);
        p = q;
    }
    const float inv = 1.f / len;
    const float ma = node(ka).m, mb = node(kb).m;
    const float La = fmaf(fa, node(ka + 1).m - ma, ma), Lb = fmaf(fb, node(kb + 1).m - mb, mb);
    const float Sm = im * inv;
    S.sm = Gj * Sm;
    S.sa = Gj * (ia * inv);
    S.sz = Gj * (ib * inv);
    const float u = ((float)ka + fa) + ls0_over;
    S.sv = Gj * fmaf(u * (Lb - La), inv, Lb - Sm);
    return S;
}

// General path of the bin means: bin j0 + 32 r + l on lane l, nodes from the
// slab when every bin of the warp has its nodes there, else from global memory.
template <int TW, int KIND>
static __device__ __noinline__ AdjSums adj_mean_general(const float2 w, const float4 g4, const TileCtx C, int lane,
                                                 const float* __restrict__ grow, float ls0_over) {
    const int c0_bi = __float_as_int(g4.x);
    const int e = rec_entry(c0_bi, C), bi = rec_bi(c0_bi);
    bool ok = C.slab_w > 0 && (unsigned)e < (unsigned)(C.pitch - 1);
    for (int o = lane; o < TW; o += 32) {
        const int j = C.j0 + o;
        if (j < C.n_lambda) {
            float fa, fb;
            const int ka = node_pos(j, bi, g4.y, g4.z, g4.w, fa) - C.klo;
            const int kb = node_pos(j + 1, bi, g4.y, g4.z, g4.w, fb) - C.klo;
            ok = ok && ka >= 0 && kb + 1 < C.slab_w;
        }
    }
    const bool use_slab = __all_sync(0xffffffffu, ok);
    AdjSums S{0.f, 0.f, 0.f, 0.f};
    for (int o = lane; o < TW; o += 32) {
        const int j = C.j0 + o;
        if (j >= C.n_lambda) break;
        const AdjSums b = adj_mean_bin<KIND>(w, g4, C, j, grow[j], use_slab, ls0_over);
        S.sm += b.sm;
        S.sa += b.sa;
        S.sz += b.sz;
        S.sv += b.sv;
    }
    return S;
}

// Kind 0 (dt/dj in (30/31, 1]): the forward's 30-bin rounds (edge l on lane l;
// see mean_rounds_near1), accumulated per entry as at bin centres.
// Lane l interpolates the cell's entries at its edge (L), takes the
// next edge's (Ln) and the enclosed node's values, and adds G_j times twice
// the entry's bin mean (U) and G_j times the entry's share of the v bracket
// (T); the weights are applied once afterwards.
template <int R>
__device__ __forceinline__ AdjSums adj_mean_near1(const float2 w, const TileCtx& C, uint32_t base, float t0, float f,
                                                  float delta, int lane, float lanef, const float (&G)[R + 1]) {
    const uint32_t p8 = (uint32_t)C.pitch * 8u, s30 = 30u * p8, s29 = 29u * p8;
    const float nld = __fmul_rn(-lanef, delta);
    const float d30 = __fmul_rn(30.f, delta);
    const float A = 1.f - delta;
    const float iA = 1.f / A;
    // absolute position of lane l's edge (node units + ls0/dls), 30 A further each round
    float u = fmaf(lanef, A, t0);
    const float du = __fmul_rn(30.f, A);
    const float2 mhalf = make_float2(-0.5f, -0.5f);
    float2 U01 = make_float2(0.f, 0.f), U23 = U01, T01 = U01, T23 = U01;
#pragma unroll
    for (int r = 0; r <= R; ++r) {
        const float g = __fadd_rn(f, nld);
        Quad Q;
        Q.a = Q.b = make_float2(0.f, 0.f);
        if (r < R || lane <= R + 1) Q = lds_quad(base, C);
        const bool up = g >= 0.f;
        const int src = up ? lane + 1 : lane - 1;
        const float2 Q01 = Q.a, Q23 = Q.b;
        const float2 X01 = make_float2(__shfl_sync(0xffffffffu, Q.a.x, src), __shfl_sync(0xffffffffu, Q.a.y, src));
        const float2 X23 = make_float2(__shfl_sync(0xffffffffu, Q.b.x, src), __shfl_sync(0xffffffffu, Q.b.y, src));
        const float2 D01 = __fadd2_rn(X01, make_float2(-Q01.x, -Q01.y));
        const float2 D23 = __fadd2_rn(X23, make_float2(-Q23.x, -Q23.y));
        const float ag = fabsf(g);
        const float2 L01 = __ffma2_rn(make_float2(ag, ag), D01, Q01);
        const float2 L23 = __ffma2_rn(make_float2(ag, ag), D23, Q23);
        const float2 N01 = make_float2(__shfl_down_sync(0xffffffffu, L01.x, 1), __shfl_down_sync(0xffffffffu, L01.y, 1));
        const float2 N23 = make_float2(__shfl_down_sync(0xffffffffu, L23.x, 1), __shfl_down_sync(0xffffffffu, L23.y, 1));
        // the node between the edges (the neighbour if g >= 0)
        const float uf = up ? 1.f : 0.f;
        const float2 K01 = __ffma2_rn(make_float2(uf, uf), D01, Q01);
        const float2 K23 = __ffma2_rn(make_float2(uf, uf), D23, Q23);
        const float ai = fmaf(-g, iA, up ? iA : 0.f);  // a / A
        const float2 dd01 = __fadd2_rn(L01, make_float2(-N01.x, -N01.y));
        const float2 dd23 = __fadd2_rn(L23, make_float2(-N23.x, -N23.y));
        // twice the bin mean: M_K + L_{l+1} + (a/A)(L - L_{l+1})
        const float2 v01 = __ffma2_rn(make_float2(ai, ai), dd01, __fadd2_rn(K01, N01));
        const float2 v23 = __ffma2_rn(make_float2(ai, ai), dd23, __fadd2_rn(K23, N23));
        const float Gj = G[r];  // 0 for lanes that own no bin of the tile
        const float2 G2 = make_float2(Gj, Gj);
        U01 = __ffma2_rn(G2, v01, U01);
        U23 = __ffma2_rn(G2, v23, U23);
        // v bracket per entry: L_{l+1} - mean - u (L - L_{l+1}) / A
        const float gu = -Gj * u * iA;
        T01 = __ffma2_rn(G2, __ffma2_rn(mhalf, v01, N01), __ffma2_rn(make_float2(gu, gu), dd01, T01));
        T23 = __ffma2_rn(G2, __ffma2_rn(mhalf, v23, N23), __ffma2_rn(make_float2(gu, gu), dd23, T23));
        if (r < R) {
            f -= d30;
            const bool carry = f < 0.f;
            f = carry ? f + 1.f : f;
            base += carry ? s29 : s30;
            u += du;
        }
    }
    return entry_sums<0>(w, 0.5f, U01, U23, T01, T23);
}

// Any dt/dj in [1/2, 2): the forward's two-read edges (mean_rounds_phi) in
// rounds of 31 bins (lane l: edge l and bin l < 31), accumulated per entry
// like adj_mean_near1: v = 2 (e_{j+1} - e_j) mean, the bracket L_{l+1} - mean +
// u (L_{l+1} - L) / (e_{j+1} - e_j). Edges are placed with all the record's
// precision, as in adj_rounds (u is a few thousand node steps).
template <int TW, int NR>
__device__ __forceinline__ AdjSums adj_mean_phi(const float2 w, const float4 g4, const TileCtx& C, int e, int bi, float A,
                                                float u0, int lane, float lanef, const float (&G)[NR]) {
    const uint32_t p8 = (uint32_t)C.pitch * 8u;
    const uint32_t base = C.slab + ((uint32_t)(bi - C.klo) * (uint32_t)C.pitch + (uint32_t)e) * 8u - kMagicBits * p8;
    const float jl = (float)C.j0 + lanef;
    float2 U01 = make_float2(0.f, 0.f), U23 = U01, T01 = U01, T23 = U01;
#pragma unroll
    for (int r = 0; r < NR; ++r) {
        const float jf = jl + 31.f * r;
        const float pp = __fmul_rn(jf, g4.z);  // exact
        const float y1 = __fadd_rd(pp, kMagic);
        const float s = __fadd_rn(pp - (y1 - kMagic), fmaf(jf, g4.w, g4.y));
        const float y = __fadd_rd(s, y1);
        const float phi = s - (y - y1);
        Quad Q, X;
        Q.a = Q.b = X.a = X.b = make_float2(0.f, 0.f);
        if (31 * r + 31 <= TW || 31 * r + lane <= TW) {  // edges 0 .. TW of the tile
            const uint32_t a = base + __float_as_uint(y) * p8;
            Q = lds_diff(a, C);
            X = lds_diff(a + p8, C);
        }
        const float d = __shfl_down_sync(0xffffffffu, y, 1) - y;  // whole nodes to edge l + 1
        const float ph1 = __shfl_down_sync(0xffffffffu, phi, 1);
        const float inv = 1.f / (d + (ph1 - phi));
        const float u = fmaf(jf, A, u0);
        const float g = lane < 31 ? G[r] : 0.f, gi = __fmul_rn(__fmul_rn(0.5f, g), lane < 31 ? inv : 0.f);
        const float gu = __fmul_rn(__fmul_rn(2.f, gi), u);
        const float2 p2 = make_float2(phi, phi), q2 = make_float2(1.f - phi, 1.f - phi);
        const float2 d2 = make_float2(d - 1.f, d - 1.f), h2 = make_float2(ph1, ph1);
        const float2 g2 = make_float2(g, g), gi2 = make_float2(gi, gi), gu2 = make_float2(gu, gu);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const float2 q = h ? Q.b : Q.a, xx = h ? X.b : X.a;
            const float2 Lv = __ffma2_rn(p2, __fadd2_rn(xx, make_float2(-q.x, -q.y)), q);
            const float2 Ln = make_float2(__shfl_down_sync(0xffffffffu, Lv.x, 1), __shfl_down_sync(0xffffffffu, Lv.y, 1));
            const float2 Mn = make_float2(__shfl_down_sync(0xffffffffu, q.x, 1), __shfl_down_sync(0xffffffffu, q.y, 1));
            const float2 v = __ffma2_rn(q2, __fadd2_rn(Lv, xx),
                                        __ffma2_rn(d2, __fadd2_rn(xx, Mn), __fmul2_rn(h2, __fadd2_rn(Mn, Ln))));
            const float2 br = __ffma2_rn(gu2, __fadd2_rn(Ln, make_float2(-Lv.x, -Lv.y)), __fmul2_rn(g2, Ln));
            float2& U = h ? U23 : U01;
            float2& T = h ? T23 : T01;
            U = __ffma2_rn(gi2, v, U);
            T = __fadd2_rn(T, __ffma2_rn(make_float2(-gi, -gi), v, br));
        }
    }
    return entry_sums<1>(w, 1.f, U01, U23, T01, T23);
}

// One particle's four sums over the tile (setup by every lane; warp-uniform path).
template <int R, int KIND, bool MEAN, int TW, int NR>
__device__ __forceinline__ AdjSums adj_particle(const float2 w, const float4 g4, const TileCtx& C, int lane,
                                                float lanef, const float (&G)[NR], const float* grow, float ls0_over) {
    const int c0_bi = __float_as_int(g4.x);
    float f;
    const int K0 = node_pos(C.j0, rec_bi(c0_bi), g4.y, g4.z, g4.w, f);  // the tile's first bin
    const int kw = K0 - C.klo;
    const float A = g4.z + g4.w;
    const int e = rec_entry(c0_bi, C);
    const bool fits = A <= C.a_max && (unsigned)kw < (unsigned)(C.slab_w - C.need) &&
                      (unsigned)e < (unsigned)(C.pitch - 1) && A > 0.f;
    const int bi = rec_bi(c0_bi);
    const float u0 = ((float)bi + g4.y) + ls0_over;
    if constexpr (KIND == 0) {
        const float delta = (1.f - g4.z) - g4.w;
        if (fits && delta >= 0.f && delta * 31.f < 1.f) {
            const uint32_t base = C.slab + ((uint32_t)(kw + lane) * (uint32_t)C.pitch + (uint32_t)e) * 8u;
            const float t0 = ((float)K0 + f) + ls0_over;
            if constexpr (MEAN) return adj_mean_near1<R>(w, C, base, t0, f, delta, lane, lanef, G);
            else return adj_near1<R>(w, C, base, t0, f, delta, lane, lanef, G);
        }
    } else if constexpr (MEAN) {
        if (fits && A >= 0.5f && A < 1.999f) return adj_mean_phi<TW, NR>(w, g4, C, e, bi, A, u0, lane, lanef, G);
    } else {
        if (fits) return adj_rounds<TW, NR>(w, g4, C, e, bi, A, u0, lanef, G);
    }
    if (!(g4.z > 0.f)) return AdjSums{0.f, 0.f, 0.f, 0.f};  // the spectrum misses every bin
    if constexpr (MEAN) return adj_mean_general<TW, KIND>(w, g4, C, lane, grow, ls0_over);
    else return adj_general<TW, KIND>(w, g4, C, lane, grow, ls0_over);
}

template <int R, int KIND, bool MEAN>
__global__ void __launch_bounds__(RUBIX_ADJ_THREADS, 1) k_adjoint_tiles(const __grid_constant__ AdjTileParams P) {
    // bins per round: kind 0 as in the forward (31; for means R rounds of 30
    // and one of R), else 32 at bin centres and 31 between 32 edges
    constexpr int TW = kind_bins(KIND) * R;
    constexpr int BR = KIND == 0 ? (MEAN ? 30 : 31) : (MEAN ? 31 : 32);
    constexpr int NR = KIND == 0 ? (MEAN ? R + 1 : R) : (TW + BR - 1) / BR;
    extern __shared__ __align__(1024) unsigned char smem[];
    uint64_t* bar = reinterpret_cast<uint64_t*>(smem);
    int* s_next = reinterpret_cast<int*>(smem + 16);
    const int lane = threadIdx.x & 31;
    const float lanef = (float)lane;
    const int nb = P.n_bands;
    const long long n_items = P.item_off[P.n_s];
    const long long n_in = P.seg_off[(long long)P.n_s * nb];
    if (n_in > P.n_cap) {
        if (blockIdx.x == 0 && threadIdx.x == 0) atomicOr(P.err, kErrBadItem);
        return;
    }
    const long long C0 = P.cost_c0;
    const long long CT = n_in + C0 * n_items;
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
    const float4* __restrict__ map4 = reinterpret_cast<const float4*>(P.map);

    for (long long t = lo / CT; t < P.n_tiles && t * CT < hi; ++t) {
        const long long a = max(lo - t * CT, 0ll), b = min(hi - t * CT, CT);
        if (a >= b) continue;
        const int ia = (int)item_lower_bound(P.items, n_items, C0, a);
        const int ib = (int)item_lower_bound(P.items, n_items, C0, b);
        const int nv = ib - ia;
        C.klo = P.tile_klo[t];
        C.j0 = (int)t * P.tile_w;
        float4* __restrict__ part = P.part + t * P.n_cap;
        for (int band = 0; band < nb; ++band) {
            C.e0 = P.band_e0[band];
            C.gband = band_ptr(P.pair, P.qdt, P.band_stride, band);
            __syncthreads();  // all warps are done with the previous slab
            if (threadIdx.x == 0) {
                *s_next = 0;
                if (C.slab_w > 0) load_slab(C, bar);
            }
            bool ok = true;
            if (C.slab_w > 0) {
                ok = mbar_wait_bounded(bar, phase, 4000000000ll);
                phase ^= 1u;
            }
            if (__syncthreads_or(!ok)) {
                if (threadIdx.x == 0) atomicOr(P.err, kErrTmaTimeout);
                return;
            }
            int v0 = 0;
            while (true) {
                const int GR = claim_size(nv - v0, RUBIX_ADJ_GRAB);
                if (lane == 0) v0 = atomicAdd(s_next, GR);
                v0 = __shfl_sync(0xffffffffu, v0, 0);
                if (v0 >= nv) break;
                int qb = 0, qe = 0, sp = 0;
                bool live = false;
                if (lane < GR && v0 + lane < nv) {
                    const Item I = P.items[ia + v0 + lane];
                    sp = I.spaxel;
                    if (sp < 0 || sp >= P.n_s) {
                        atomicOr(P.err, kErrBadItem);
                    } else {
                        qb = max(I.begin, P.seg_off[(long long)sp * nb + band]);
                        qe = min(I.end, P.seg_off[(long long)sp * nb + band + 1]);
                        live = qb < qe;
                        // the item's first weights and record, on their way to L1,
                        // and its tile slice of dL/dcube0 on its way to L2
                        if (live) {
                            asm volatile("prefetch.global.L1 [%0];" ::"l"(P.wu + qb));
                            asm volatile("prefetch.global.L1 [%0];" ::"l"(map4 + qb));
                            const float* gs = P.G0 + (long long)sp * P.n_lambda + C.j0;
                            const int nbin = min(P.tile_w + 1, P.n_lambda - C.j0);
#pragma unroll 1
                            for (int o = 0; o < nbin; o += 32)
                                asm volatile("prefetch.global.L2 [%0];" ::"l"(gs + o));
                        }
                    }
                }
                unsigned m = __ballot_sync(0xffffffffu, live);
                while (m) {
                    const int src = __ffs(m) - 1;
                    m &= m - 1;
                    const int q0 = __shfl_sync(0xffffffffu, qb, src);
                    const int q1 = __shfl_sync(0xffffffffu, qe, src);
                    const int s = __shfl_sync(0xffffffffu, sp, src);
                    // this tile's slice of the spaxel's dL/dcube0 row, one bin per lane and round
                    float G[NR];
                    const float* __restrict__ grow = P.G0 + (long long)s * P.n_lambda;
#pragma unroll
                    for (int r = 0; r < NR; ++r) {
                        const int o = BR * r + lane;
                        G[r] = (lane < BR && o < TW && C.j0 + o < P.n_lambda) ? grow[C.j0 + o] : 0.f;
                    }
                    for (int q = q0; q < q1; ++q) {
                        if (q + 1 < q1) {
                            asm volatile("prefetch.global.L1 [%0];" ::"l"(P.wu + q + 1));
                            asm volatile("prefetch.global.L1 [%0];" ::"l"(map4 + q + 1));
                        }
                        const AdjSums S = adj_particle<R, KIND, MEAN, TW, NR>(P.wu[q], map4[q], C, lane, lanef,
                                                                              G, grow, P.ls0_over);
                        // the four sums over the warp with 6 shuffles: halves of the
                        // warp trade pairs, quarters trade singles, then a butterfly
                        // over 8 lanes; lane 8 v ends with sum v (v = sm, sa, sz, sv)
                        const bool hi16 = lane >= 16, hi8 = (lane & 8) != 0;
                        const float r0 = __shfl_xor_sync(0xffffffffu, hi16 ? S.sm : S.sz, 16);
                        const float r1 = __shfl_xor_sync(0xffffffffu, hi16 ? S.sa : S.sv, 16);
                        const float b0 = (hi16 ? S.sz : S.sm) + r0, b1 = (hi16 ? S.sv : S.sa) + r1;
                        float c = (hi8 ? b1 : b0) + __shfl_xor_sync(0xffffffffu, hi8 ? b0 : b1, 8);
#pragma unroll
                        for (int o = 4; o > 0; o >>= 1) c += __shfl_xor_sync(0xffffffffu, c, o);
#if RUBIX_DEBUG
                        dbg_check(q >= 0 && q < P.n_cap, P.err);
#endif
                        if ((lane & 7) == 0) reinterpret_cast<float*>(part + q)[lane >> 3] = c;
                    }
                }
            }
        }
    }
}

typedef void (*AdjointFn)(const AdjTileParams);
template <int KIND>
AdjointFn adjoint_fn(int R, bool mean) {
    switch (R) {
#define RUBIX_ADJ_R(r) \
    case r: return mean ? k_adjoint_tiles<r, KIND, true> : k_adjoint_tiles<r, KIND, false>;
        RUBIX_ROUNDS(RUBIX_ADJ_R)
#undef RUBIX_ADJ_R
        default: return nullptr;
    }
}
AdjointFn adjoint_fn_k0(int R, bool mean);
AdjointFn adjoint_fn_k1(int R, bool mean);
AdjointFn adjoint_fn_k2(int R, bool mean);

}  // namespace rubix
