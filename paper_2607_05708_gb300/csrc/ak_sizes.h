// Scratch sizes of the prefix sum and of the radix sort (ak_graph.cu).  Plain
// C++, so that they can be checked without a GPU.
//
// A scratch is often sized once for several sorts, by the largest count, so
// neither size may fall as n grows.
#pragma once

#include <stddef.h>
#include <stdint.h>

namespace ak {

constexpr int SCAN_TILE = 2048;         // values a CTA scans
constexpr int RS_TILE = 4096;           // pairs a CTA sorts
constexpr int RS_SMALL_TILE = 1024;     // the same of a small sort,
constexpr int64_t RS_SMALL_TILES = 256; // of at most this many tiles

inline size_t scan_tmp_bytes(int64_t n) {
    size_t tot = 0;
    int64_t m = n;
    do {
        const int64_t tiles = (m + SCAN_TILE - 1) / SCAN_TILE;
        tot += (size_t)(2 * tiles + 2) * sizeof(int64_t);
        m = tiles;
    } while (m > 1);
    return tot + 64;
}

// The large sort's 64-bit histograms, their scan and its scratch; the small
// sort's three 32-bit histograms, which take three times the bytes a pair and so
// still count (at their largest) where a sort is too long for them.
inline size_t radix_tmp_bytes(int64_t n) {
    const int64_t m = 256 * ((n + RS_TILE - 1) / RS_TILE);
    const size_t big = (size_t)(2 * m + 1) * sizeof(int64_t) + scan_tmp_bytes(m) + 256;
    const int64_t st = (n + RS_SMALL_TILE - 1) / RS_SMALL_TILE;
    const size_t small =
        (size_t)3 * 256 * (st < RS_SMALL_TILES ? st : RS_SMALL_TILES) * sizeof(int) + 256;
    return big > small ? big : small;
}

}  // namespace ak
