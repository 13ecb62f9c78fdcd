// sort_layout.h -- tiles and scratch of the radix sort (sort.cu): host
// arithmetic without a GPU, so that the sizing rule can be checked on its own.
#pragma once

#include <stddef.h>
#include <stdint.h>

#include <algorithm>

namespace rubix {

constexpr int kSortThreads = 256;
constexpr int kMaxBuckets = 512;   // up to 9 bits per pass
constexpr int kScanTile = 4096;    // digit counts per tile of the scan

// Words of a chained scan's state (common.cuh): the ticket and a word per tile.
inline size_t chain_words(long long tiles) { return (size_t)tiles + 1; }

// Keys per tile: 16 per thread, or 4 while that leaves the tiles fewer than two
// per SM (each round of a tile is a dependent step: 1e4 keys took 10 us for the
// counts and 14 us for the scatter in 3 tiles of 4096).
constexpr int kRoundsLong = 16, kRoundsShort = 4;
inline long long short_tile_keys(int n_sm) { return 2ll * n_sm * kSortThreads * kRoundsLong; }  // the most of them

struct SortLayout {
    int rounds;           // keys per thread of a tile
    int n_tiles;
    int passes, bits;     // digits of bits / passes bits, rounded up
    long long n_counts;   // digit counts of a pass
    size_t ints;          // scratch: one int to align, the scan's chain, counts and offsets
};

// Sort of n keys in [0, n_keys) (long_tiles: the large tiles whatever n is).
inline SortLayout sort_layout(long long n, int n_keys, int n_sm, bool long_tiles) {
    SortLayout L;
    L.bits = 1;
    while ((1ll << L.bits) < (long long)n_keys) ++L.bits;
    L.passes = (L.bits + 8) / 9;
    const int per = (L.bits + L.passes - 1) / L.passes;
    L.rounds = long_tiles || n > short_tile_keys(n_sm) ? kRoundsLong : kRoundsShort;
    const long long tile = (long long)kSortThreads * L.rounds;
    L.n_tiles = (int)((n + tile - 1) / tile);
    L.n_counts = (long long)L.n_tiles << per;
    L.ints = 1 + 2 * chain_words((L.n_counts + kScanTile - 1) / kScanTile) + 2 * (size_t)L.n_counts;
    return L;
}

// Scratch for every sort of at most n keys, of any width. Not the layout of n
// alone: at the switch to long tiles the need drops to a quarter, so that a call
// below it can need more than the capacity does.
inline size_t sort_scratch_ints(long long n, int n_sm, bool long_tiles) {
    const int nine_bits = 1 << 9;
    const size_t own = sort_layout(n, nine_bits, n_sm, long_tiles).ints;
    return std::max(own, sort_layout(std::min(n, short_tile_keys(n_sm)), nine_bits, n_sm, long_tiles).ints);
}

}  // namespace rubix
