// common.cuh -- internal helpers shared by the library's kernels (not part of the ABI).
#pragma once

#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

namespace rubix {

constexpr double kC_kms = 299792.458;

// Error word written by kernels (bit flags), read by the host after a forward.
enum DeviceError : unsigned {
    kErrTmaTimeout = 1u,      // a bounded wait expired (the mbarrier of a slab or cube row load, the items' scan)
    kErrBadItem = 2u,         // a work item pointed outside its buffers
    kErrBounds = 4u,          // debug builds: a computed index fell outside its buffer
};

// Debug builds (RUBIX_DEBUG=1, a separate library built by the tests) check
// the shared-memory and record indices the deposit and the adjoint compute
// against their buffers and set kErrBounds instead of faulting; release
// builds compile none of it.
#ifndef RUBIX_DEBUG
#define RUBIX_DEBUG 0
#endif
__device__ __forceinline__ void dbg_check(bool ok, unsigned* err) {
#if RUBIX_DEBUG
    if (!ok && err) atomicOr(err, kErrBounds);
#else
    (void)ok;
    (void)err;
#endif
}

// ----------------------------------------------------------------------------
// Shared-memory barrier and TMA (inline PTX, sm_90+ forms valid on sm_103a)
// ----------------------------------------------------------------------------
__device__ __forceinline__ uint32_t smem_addr(const void* p) {
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_addr(bar)), "r"(count) : "memory");
}

__device__ __forceinline__ void fence_mbar_init() {
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

__device__ __forceinline__ void fence_proxy_async_smem() {
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

__device__ __forceinline__ void mbar_arrive_expect_tx(uint64_t* bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(bar)), "r"(bytes)
                 : "memory");
}

// Bounded wait on phase `parity` of an mbarrier. Returns false if it did not
// complete within ~max_cycles SM clocks (the caller records an error and
// stops using the buffer instead of spinning forever).
__device__ __forceinline__ bool mbar_wait_bounded(uint64_t* bar, uint32_t parity, long long max_cycles) {
    const uint32_t a = smem_addr(bar);
    auto done = [&]() {
        uint32_t d;
        asm volatile(
            "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
            : "=r"(d)
            : "r"(a), "r"(parity)
            : "memory");
        return d != 0;
    };
    if (done()) return true;  // (no clock read when the data is there)
    const long long t0 = clock64();
    while (!done())
        if (clock64() - t0 > max_cycles) return false;
    return true;
}

// Bulk copy of `bytes` (a multiple of 16, both addresses 16-byte aligned) from
// global memory to the shared-space address dst.
__device__ __forceinline__ void bulk_load(uint32_t dst, const void* src, uint32_t bytes, uint64_t* bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
                 "l"(src), "r"(bytes), "r"(smem_addr(bar))
                 : "memory");
}

__device__ __forceinline__ void sts_f4(uint32_t dst, float x, float y, float z, float w) {
    asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(dst), "f"(x), "f"(y), "f"(z), "f"(w) : "memory");
}

// 3-D tiled TMA load (c0 innermost).
__device__ __forceinline__ void tma_load_3d(void* smem_dst, const CUtensorMap* map, uint64_t* bar, int c0, int c1,
                                            int c2) {
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5}], "
        "[%2];" ::"r"(smem_addr(smem_dst)),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(smem_addr(bar)), "r"(c0), "r"(c1), "r"(c2)
        : "memory");
}

// ----------------------------------------------------------------------------
// Philox4x32-10 (Salmon, Moraes, Dror, Shaw, SC'11), written from the
// published round function: two 32x32->64 multiplies per round with the
// multipliers 0xD2511F53 / 0xCD9E8D57 and Weyl key increments 0x9E3779B9 /
// 0xBB67AE85.
// ----------------------------------------------------------------------------
struct U4 { uint32_t x, y, z, w; };

__host__ __device__ __forceinline__ U4 philox4x32_10(U4 ctr, uint32_t k0, uint32_t k1) {
    const uint32_t M0 = 0xD2511F53u, M1 = 0xCD9E8D57u, W0 = 0x9E3779B9u, W1 = 0xBB67AE85u;
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        uint64_t p0 = (uint64_t)M0 * ctr.x;
        uint64_t p1 = (uint64_t)M1 * ctr.z;
        uint32_t hi0 = (uint32_t)(p0 >> 32), lo0 = (uint32_t)p0;
        uint32_t hi1 = (uint32_t)(p1 >> 32), lo1 = (uint32_t)p1;
        U4 n;
        n.x = hi1 ^ ctr.y ^ k0;
        n.y = lo1;
        n.z = hi0 ^ ctr.w ^ k1;
        n.w = lo0;
        ctr = n;
        k0 += W0;
        k1 += W1;
    }
    return ctr;
}

// ----------------------------------------------------------------------------
// SSP cell search: half-open cell [node_i, node_i+1) holding q, clamped outside
// the grid (t = 0 below the first node, t = 1 at or above the last); dt = dt/dq
// inside the grid, 0 when clamped. Shared by the key, setup and adjoint kernels
// so that they always agree on the cell of a particle.
// ----------------------------------------------------------------------------
__device__ __forceinline__ void ssp_cell(float q, const float* __restrict__ nodes, int n, int& i, float& t,
                                         float& dt) {
    if (n < 2 || !(q > nodes[0])) { i = 0; t = 0.f; dt = 0.f; return; }
    if (q >= nodes[n - 1]) { i = n - 2; t = 1.f; dt = 0.f; return; }
    int lo = 0, hi = n - 1;  // nodes[lo] <= q < nodes[hi]
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (nodes[mid] <= q) lo = mid; else hi = mid;
    }
    i = lo;
    const float h = nodes[lo + 1] - nodes[lo];
    t = (q - nodes[lo]) / h;
    dt = 1.f / h;
}

// Age band of an age cell: the template grid is split into n_bands groups of
// `apb` age cells so that one band's templates fit a wide shared-memory slab.
__device__ __forceinline__ int age_band(int ia, int apb, int n_bands) {
    const int b = (apb > 0) ? ia / apb : 0;
    return b < n_bands - 1 ? b : n_bands - 1;
}

// ----------------------------------------------------------------------------
// Scans in one launch. Blocks take tiles in order from a ticket, publish their
// tile's sum, and add up the sums published before theirs: a block waits only
// for blocks that hold an earlier ticket, which are running and publish without
// waiting for anyone. chain[0] is the ticket, chain[1 + tile] the tile's sum
// with its top bit set; all are cleared beforehand. The wait has a limit in cycles
// (the blocks of a GPU that was taken away from the process in between may meet
// it), after which the prefix says that sums are missing from it: kChainShort, a
// millisecond, where the block can then do without them, kChainLong where that is
// an error. (chain_words in sort_layout.h gives the words of a chain.)
// ----------------------------------------------------------------------------
struct ChainShared {
    unsigned ticket;
    unsigned long long warp[32];
    unsigned long long total;
};

__device__ __forceinline__ unsigned chain_ticket(unsigned long long* chain, ChainShared& sh) {
    if (threadIdx.x == 0) sh.ticket = (unsigned)atomicAdd(chain, 1ull);
    __syncthreads();
    return sh.ticket;
}

// Sum over the block (all threads take part; up to 1024 threads).
__device__ __forceinline__ unsigned long long block_exclusive(unsigned long long v, ChainShared& sh,
                                                              unsigned long long& total) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    unsigned long long x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned long long y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) sh.warp[wid] = x;
    __syncthreads();
    if (wid == 0) {
        const unsigned long long t = (lane < (int)((blockDim.x + 31) >> 5)) ? sh.warp[lane] : 0ull;
        unsigned long long s = t;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned long long y = __shfl_up_sync(0xffffffffu, s, o);
            if (lane >= o) s += y;
        }
        sh.warp[lane] = s - t;
        if (lane == 31) sh.total = s;
    }
    __syncthreads();
    const unsigned long long r = x - v + sh.warp[wid];
    total = sh.total;
    __syncthreads();
    return r;
}

constexpr long long kChainShort = 2000000ll, kChainLong = 4000000000ll;
constexpr unsigned long long kChainMissing = 1ull << 52;

// Exclusive prefix of v over all threads of all tiles before this one (sums below
// 2^52); at least kChainMissing, for every thread of the block, if a wait ran out:
// its lower bits are then a sum too small, never too large. quiet (tests): nothing
// is published, and waits are short.
__device__ __forceinline__ unsigned long long chain_exclusive(unsigned long long v, unsigned tile,
                                                              unsigned long long* chain, ChainShared& sh, long long wait,
                                                              bool quiet) {
    unsigned long long total;
    const unsigned long long e = block_exclusive(v, sh, total);
    volatile unsigned long long* pub = chain + 1;
    if (threadIdx.x == 0 && !quiet) pub[tile] = total | (1ull << 63);
    unsigned long long before = 0;
    if (quiet) wait = kChainShort;
    const long long t0 = clock64();
    for (unsigned i = threadIdx.x; i < tile; i += blockDim.x) {
        unsigned long long w = pub[i];
        while (!(w >> 63) && clock64() - t0 < wait) w = pub[i];
        before += (w >> 63) ? w & ~(1ull << 63) : kChainMissing;
    }
    unsigned long long sum;
    block_exclusive(before, sh, sum);
    return sum + e;
}

// ----------------------------------------------------------------------------
// Work descriptors
// ----------------------------------------------------------------------------
// Per in-field particle, in sorted order: everything the deposit's fast rounds
// need (32 B). With t(j) = tau(j) + s(j), tau the node position of bin j for a
// particle at rest, s(j) = s0 + (j - jc) g is the particle's Doppler shift in
// nodes, in fixed point: s0 in units of 2^-fb nodes, g of 2^-(fb + 13)
// (SlabParams::fb, jc), so that a tile's first node and fraction are one
// multiply-high and an addition to the tile's constant.
struct __align__(16) DepRec {
    float w[4];        // mass * flux_scale * bilinear weights: (ia,iz) (ia+1,iz) (ia,iz+1) (ia+1,iz+1)
    int s0;            // s(jc)
    int g;             // ds/dj
    float d;           // kind 0: 1 - dt/dj; kinds 1, 2: dt/dj less that of a particle at rest
    unsigned ef;       // 8 * (entry of the cell within its band) | RecPath << 30
};
static_assert(sizeof(DepRec) == 32, "DepRec layout");

// Which rounds a particle takes in every tile: the kind's own, the two-read
// rounds (centres) or two-read edges (means), or the per-bin path.
enum RecPath : unsigned { kPathMain = 0u, kPathTwoRead = 1u, kPathBins = 2u };

// Smallest 1 - dt/dj of the kind-1 rounds (deposit_kernel.cuh).
constexpr float kShuffleTol = 1e-5f;

// The full affine map of the same particle (16 B), for the per-bin path and the
// adjoint: bin j at fractional SSP node position t(j) = bi + bf + j*(a_hi +
// a_lo). a_hi keeps 11 significant bits, so j*a_hi is exact in FP32 for
// j < 2^13 and only the small term j*a_lo is rounded.
struct __align__(16) MapRec {
    int c0_bi;         // (SSP cell ia * n_Z + iz) << 16 | (floor(t(0)) & 0xffff)
    float bf;          // t(0) - floor(t(0)), in [0, 1)
    float a_hi;        // dt/dj, high part (0: the spectrum misses every output bin)
    float a_lo;        // dt/dj, low part
};
static_assert(sizeof(MapRec) == 16, "MapRec layout");

__device__ __forceinline__ int rec_c0(int c0_bi) { return (int)((unsigned)c0_bi >> 16); }
__device__ __forceinline__ int rec_bi(int c0_bi) { return (c0_bi << 16) >> 16; }

// Per in-field particle, sorted order: the inputs of its spectrum, kept for backward.
struct __align__(16) PartRec {
    float mass, age, Z, v;
};

// One unit of deposit work: particles [begin, end) of spaxel `spaxel`,
// written to the cube row (part_row < 0) or to partial row `part_row`.
struct __align__(16) Item {
    int spaxel;
    int begin;
    int end;
    int part_row;
};

}  // namespace rubix
