// tile.cuh -- device helpers shared by the deposit (K4) and the adjoint over
// the same (wavelength tile, work item, age band) decomposition: work-item
// search over the cost space, the bin -> SSP node map, and the template slab.
#pragma once

#include <climits>

#include "common.cuh"
#include "kernels.h"

namespace rubix {

// First item index i in [0, n] with items[i].begin + c0 * i >= x (item n is
// the virtual end).
__device__ __forceinline__ long long item_lower_bound(const Item* __restrict__ items, long long n, long long c0,
                                                      long long x) {
    long long lo = 0, hi = n;
    while (lo < hi) {
        const long long mid = (lo + hi) >> 1;
        const long long pre = (long long)items[mid].begin + c0 * mid;
        if (pre < x) lo = mid + 1; else hi = mid;
    }
    return lo;
}

// Node position of output bin j: t(j) = K + phi, phi in [0, 1). j*a_hi is
// exact in FP32; only the small j*a_lo term is rounded.
__device__ __forceinline__ int node_pos(int j, int bi, float bf, float a_hi, float a_lo, float& phi) {
    const float jf = (float)j;
    const float pp = jf * a_hi;
    const float pi = floorf(pp);
    const float s = (pp - pi) + fmaf(jf, a_lo, bf);
    const float fl = floorf(s);
    phi = s - fl;
    return bi + (int)pi + (int)fl;
}

struct TileCtx {
    int j0, klo, slab_w, pitch, e0, es, n_lambda, n_ls, pad;
    uint32_t slab;         // shared-space address of the slab
    const void* gband;     // this band's entries in global memory (FP32 float2 or 16-bit uint32_t)
    int qdt;               // 0: FP32, 1: BF16, 2: FP16
    float a_max;           // largest dt/dj whose rounds stay within `need` nodes (adjoint)
    int need;              // nodes the rounds of one particle can read, from its first (adjoint)
#if RUBIX_DEBUG
    unsigned* err;         // error word for the debug build's index checks
#endif
};

// Entry of a record's cell within the band's node rows (es = 2 for a grid of
// one metallicity, whose rows repeat each age's entry).
__device__ __forceinline__ int rec_entry(int c0_bi, const TileCtx& C) { return rec_c0(c0_bi) * C.es - C.e0; }

// The two 16-bit values of an entry as FP32 (exact).
__device__ __forceinline__ float2 unpack_pair(uint32_t v, int qdt) {
    if (qdt == 1) return make_float2(__uint_as_float(v << 16), __uint_as_float(v & 0xffff0000u));
    return make_float2(__half2float(__ushort_as_half((unsigned short)(v & 0xffffu))),
                       __half2float(__ushort_as_half((unsigned short)(v >> 16))));
}

// A cell's two entries (four corner templates) at one node.
struct Quad {
    float2 a, b;  // corners (ia, iz) (ia+1, iz); (ia, iz+1) (ia+1, iz+1)
};

// Shared-memory read of the two entries at byte address `addr`. Two 8-byte
// loads: 32 lanes on consecutive nodes are an odd number of 8-byte entries
// apart, so each load is conflict-free (two wavefronts).
__device__ __forceinline__ Quad lds_quad(uint32_t addr, const TileCtx& C) {
    Quad q;
#if RUBIX_DEBUG
    const uint32_t off = addr - C.slab;
    const bool ok = off + 16u <= (uint32_t)(C.slab_w * C.pitch) * 8u && (off & 7u) == 0u;
    dbg_check(ok, C.err);
    if (!ok) {
        q.a = q.b = make_float2(0.f, 0.f);
        return q;
    }
#endif
    asm volatile("ld.shared.v2.f32 {%0, %1}, [%2];" : "=f"(q.a.x), "=f"(q.a.y) : "r"(addr));
    asm volatile("ld.shared.v2.f32 {%0, %1}, [%2+8];" : "=f"(q.b.x), "=f"(q.b.y) : "r"(addr));
    return q;
}

// The same from the band's global array (zero outside the template range: the
// template's zero extension). e: the cell's entry within the band.
__device__ __forceinline__ Quad quad_global(const TileCtx& C, int e, int k) {
    Quad q;
    if (k < 0 || k >= C.n_ls) {
        q.a = q.b = make_float2(0.f, 0.f);
        return q;
    }
    const long long i = (long long)(k + C.pad) * C.pitch + e;
    if (C.qdt) {
        const uint32_t* g = static_cast<const uint32_t*>(C.gband) + i;
        q.a = unpack_pair(__ldg(g), C.qdt);
        q.b = unpack_pair(__ldg(g + 1), C.qdt);
    } else {
        const float2* g = static_cast<const float2*>(C.gband) + i;
        q.a = __ldg(g);
        q.b = __ldg(g + 1);
    }
    return q;
}

// Node k of a cell from the slab or, with use_slab false, from global memory.
__device__ __forceinline__ Quad quad_at(const TileCtx& C, bool use_slab, int e, int k) {
    return use_slab ? lds_quad(C.slab + (uint32_t)((k - C.klo) * C.pitch + e) * 8u, C) : quad_global(C, e, k);
}

// First row of a slab in the band's padded array. A slab that lies outside the
// templates altogether is zero wherever it is read from.
__device__ __forceinline__ int slab_row(const TileCtx& C) {
    return max(-C.slab_w, min(C.klo, (C.n_ls + 3) / 4 * 4)) + C.pad;
}

// Slab of a (tile, band) by bulk copies (FP32): the band's entries are stored
// contiguously, node rows padded with zero nodes on both sides, so the slab is
// one contiguous range, taken in pieces. Issued by one thread; `bar` gets the
// bytes. klo is a multiple of 4: 16-byte aligned.
__device__ __forceinline__ void load_slab(const TileCtx& C, uint64_t* bar) {
    const uint32_t bytes = (uint32_t)(C.slab_w * C.pitch) * 8u;
    const char* src = static_cast<const char*>(C.gband) + (long long)slab_row(C) * C.pitch * 8;
    fence_proxy_async_smem();
    mbar_arrive_expect_tx(bar, bytes);
    for (uint32_t o = 0; o < bytes; o += 16384u) bulk_load(C.slab + o, src + o, min(16384u, bytes - o), bar);
}

// Slab of a (tile, band) from 16-bit entries, by all threads of the CTA: the
// same contiguous range read in 16-byte pieces (four entries), widened to
// FP32; kFill loads are in flight per thread before their stores. The caller
// synchronises the CTA afterwards.
__device__ __forceinline__ void fill_slab16(const TileCtx& C) {
    constexpr int kFill = 4;
    const int T = blockDim.x, total = C.slab_w * C.pitch / 4;  // slab_w is a multiple of 4
    const uint4* src = reinterpret_cast<const uint4*>(static_cast<const uint32_t*>(C.gband) +
                                                      (long long)slab_row(C) * C.pitch);
    for (int i0 = threadIdx.x; i0 < total; i0 += kFill * T) {
        uint4 v[kFill];
#pragma unroll
        for (int u = 0; u < kFill; ++u) v[u] = i0 + u * T < total ? __ldg(src + i0 + u * T) : make_uint4(0, 0, 0, 0);
#pragma unroll
        for (int u = 0; u < kFill; ++u) {
            const int i = i0 + u * T;
            if (i < total) {
                const float2 x = unpack_pair(v[u].x, C.qdt), y = unpack_pair(v[u].y, C.qdt);
                const float2 z = unpack_pair(v[u].z, C.qdt), w = unpack_pair(v[u].w, C.qdt);
                sts_f4(C.slab + (uint32_t)i * 32u, x.x, x.y, y.x, y.y);
                sts_f4(C.slab + (uint32_t)i * 32u + 16u, z.x, z.y, w.x, w.y);
            }
        }
    }
}

// Work items a warp claims at once with `left` of the band's still to claim:
// `most` while every warp has plenty, then two, one at a time at the end, where
// the band's barrier waits for the last warp (claims of four throughout: 3.41 ms
// on the mid-size galaxy against 3.27, and 25 of a CTA's warps idle on a galaxy
// of 1e4 particles; of two throughout: 53.96 ms on the large galaxy against 53.6,
// where each claim's look-up chain counts).
__device__ __forceinline__ int claim_size(int left, int most) {
    const int nw = (int)(blockDim.x >> 5);
    return left > 40 * nw ? most : (left > 2 * nw ? 2 : 1);
}

// Mass-weighted bilinear template value at one node: sum_c w_c q_c.
__device__ __forceinline__ float quad_dot(const float4 w, const Quad& q) {
    float2 p = __fmul2_rn(make_float2(w.x, w.y), q.a);
    p = __ffma2_rn(make_float2(w.z, w.w), q.b, p);
    return p.x + p.y;
}

// ----------------------------------------------------------------------------
// Node positions of a particle's rounds without a chain from round to round.
// Adding a value x in (-2^21, 2^21) to kMagic with rounding towards minus
// infinity gives kMagic + floor(x) exactly, whose low mantissa bits are the
// integer: one addition floors, and the address is one integer multiply-add of
// those bits.
// ----------------------------------------------------------------------------
constexpr float kMagic = 12582912.f;          // 1.5 * 2^23
constexpr uint32_t kMagicBits = 0x4b400000u;  // its bit pattern

// Per-lane position of the rounds of kBins bins: bin j0 + kBins r + lane sits
// at node K0 + il + r ib + x_r with x_r = x0 + r fb, where il and ib are the
// whole nodes of lane (kBins) bins at rest, the same for every particle, so
// that x_r stays below a few and keeps FP32's absolute precision however wide
// the tile.
struct LanePos {
    float x0, fb;
    uint32_t base;  // byte address of node K0 + il of the cell, less kMagicBits nodes
    float nf;       // K0 + il - klo
};

// first index i in [0, n] with v[i] > x  (v non-decreasing)
__device__ __forceinline__ int upper_bound_ll(const long long* __restrict__ v, int n, long long x) {
    int lo = 0, hi = n;
    while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (v[mid] <= x) lo = mid + 1; else hi = mid;
    }
    return lo;
}

}  // namespace rubix
