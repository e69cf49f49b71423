// radix_geom.cuh -- tiling of the radix sort and the size of its count buffer.
// Plain C++ apart from the device-side count, so that the sizes can be checked
// on the host.
#pragma once
#include <stdint.h>

#ifdef __CUDACC__
#define SPH_HD __host__ __device__
#else
#define SPH_HD
#endif

namespace sph {

constexpr int kRadixThreads = 256;                  // threads per block, one digit each
constexpr int kRadixItems = 8;                      // keys per thread in the sort
constexpr int kRadixItemsSmall = 2;                 // ... of at most kRadixSmallN keys
constexpr int64_t kRadixSmallN = 262144;

// Tiling of the radix sort, and the digit counts of one of its passes: per
// tile [tiles][256], then per group of 2^group_shift tiles [groups][256].
struct RadixGeom {
    bool chained;  // each pass counts for the next (else a histogram kernel does)
    int items, tiles, groups, tile_shift, group_shift;
    SPH_HD int64_t counts() const { return (int64_t)(tiles + groups) * 256; }
#ifdef __CUDACC__
    // c keys of tile t have `digit`
    __device__ __forceinline__ void count(uint32_t* hist, int64_t t, uint32_t digit,
                                          uint32_t c) const {
        if (c == 0) return;
        atomicAdd(&hist[t * 256 + digit], c);
        if (groups > 1)
            atomicAdd(&hist[((int64_t)tiles + (t >> group_shift)) * 256 + digit], c);
    }
#endif
};

// Tiles of the sort for nt keys. Up to kRadixSmallN a chained sort with tiles
// of 512 keys, so that there are blocks enough for the chip; beyond, where its
// additions contend, a histogram kernel per pass and tiles of 2048. The line is
// where the two cross. Cells phase (bounding box to permute) of a patch in us,
// chained / with histograms: 4,096 keys 42 / 56, 27,000 52 / 66, 104k 73 / 85,
// 195k 92 / 100, 262k 101 / 100, 301k 111 / 108, 405k 136 / 125, 1M 269 / 210; of
// a sphere 200k 96 / 105, 262k 106 / 105, 300k 117 / 114.
inline RadixGeom radix_geom(int64_t nt) {
    RadixGeom R;
    R.chained = nt <= kRadixSmallN;
    R.items = R.chained ? kRadixItemsSmall : kRadixItems;
    const int64_t tile = (int64_t)kRadixThreads * R.items;
    R.tile_shift = 0;
    while ((int64_t)1 << R.tile_shift < tile) R.tile_shift += 1;
    R.tiles = (int)((nt + tile - 1) / tile);
    // up to 64 tiles: a block reads the counts of every tile; more: groups of
    // about sqrt(tiles), one count per group and one per earlier tile of its own
    R.group_shift = 4;
    while (((int64_t)4 << (2 * R.group_shift)) < R.tiles) R.group_shift += 1;
    if (R.tiles <= 64) R.group_shift = 6;
    R.groups = ((R.tiles - 1) >> R.group_shift) + 1;
    return R;
}

// Counts of one pass for any sort of at most n keys. counts() does not grow
// steadily with the keys: where group_shift steps up (1,024 to 1,025 tiles) the
// groups halve, and a context of slightly more than that needs the counts of
// the smaller sort. So the size comes from a bound that does: the groups are
// at least 16 tiles each beyond 64 tiles and one below, at most tiles / 16 + 1
// of them either way.
inline int64_t radix_counts(int64_t n) {
    auto bound = [](int64_t tiles) { return (tiles + tiles / 16 + 1) * 256; };
    const int64_t small = bound(radix_geom(n < kRadixSmallN ? n : kRadixSmallN).tiles);
    const int64_t all = bound(radix_geom(n).tiles);
    return small > all ? small : all;
}

}  // namespace sph
