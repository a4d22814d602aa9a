// How a decode step over a bf16 or 4-bit cache is spread over the device (host;
// no CUDA): the thread blocks of a (request, KV head) pair and, in batches of
// unequal requests, the parts a pair is cut into.
#pragma once
#include <stdint.h>

#include <algorithm>

#ifndef VC_HD
#ifdef __CUDACC__
#define VC_HD __host__ __device__ __forceinline__
#else
#define VC_HD inline
#endif
#endif

namespace vc {

constexpr int kTileKeys = 32;                  // keys per tile (one key group of the 4-bit form)
constexpr int kDecTileWarps = 4;               // warps per CTA, a tile each at a time

// Cluster sizes decode_tiles_kernel is launched with.
constexpr int kClusterSizes[] = {1, 2, 3, 4, 5, 6, 7, 8, 12, 16};
constexpr int kClusterKinds = (int)(sizeof(kClusterSizes) / sizeof(int));

// How many clusters of each size fit on a device at once (0: not launchable).
struct DecodeFit {
  int n[kClusterKinds] = {};
};

// Tiles of a request: visual and text rows in tiles of their own.
inline int64_t decode_tiles(int64_t B, int64_t T) {
  return (B + kTileKeys - 1) / kTileKeys + (T + kTileKeys - 1) / kTileKeys;
}

struct DecodePlan {
  int cluster;         // CTAs per pair
  int part_tiles;      // > 0: CTAs of their own (cluster 1) for every part of at most this many tiles
};

// Parts of a pair of `tiles` tiles (a pair without keys is one), and the tiles of
// each: equal, whole rounds of the CTA's warps.
inline int decode_parts(int64_t tiles, int part_tiles) {
  return (int)std::max<int64_t>(1, (tiles + part_tiles - 1) / part_tiles);
}
VC_HD int decode_tiles_per_part(int tiles, int parts) {
  const int per = (tiles + parts - 1) / parts;
  return (per + kDecTileWarps - 1) / kDecTileWarps * kDecTileWarps;
}

// One cluster a pair, no parts: the smallest cluster that gives every warp at
// most one tile, or else the largest with which all pairs are on the device at
// once (measured: one request, 137 tiles a pair, 10.4 us a layer with 4
// CTAs, 7.0 with 8, 5.7 with 16; 16 requests 24.0 to 24.3 us with 2 or 4 CTAs
// a pair and 28.5 with 6, which no longer fit at once).
//
// All pairs then get as many warps, so where one request is far longer than the
// others its warps run on alone, a tile in 0.78 us (4-bit: 1.15): 64 requests of
// 21 tiles, one with 512 text tiles more, took 104 us a layer for 0.12 GB.  With
// work for every warp the memory allows a tile in 2.8 us (4-bit: 1.6).  So where
// the longest pair has more than kEvenCost times the tiles a warp of an even
// spread and kPartCost beyond that (what the second kernel and its launch cost),
// the pairs are cut into parts, which a second kernel merges.  One rule for both
// forms, whose bits must agree; measured, us a layer (one cluster a pair | parts;
// 4-bit): that batch 104 | 31 (153 | 31); 32 requests of 200 to 6,400 rows 30 | 26
// (55 | 31); 12 requests, one of 12,000 rows 21 | 14 (34 | 18); 1 of 32,768 rows
// 15 | 24 (26 | 28); 64 requests, half with 8,192 text rows 91 | 96 (102 | 95).
constexpr int kEvenCost = 2, kPartCost = 10;
constexpr int kPartMin = 4, kPartMax = 16;     // tiles a warp of a part
constexpr int kPartsMax = 256;                 // parts of a pair

// tiles[r]: decode_tiles of request r.
inline DecodePlan plan_decode(const int64_t* tiles, int n_req, int Hkv, const DecodeFit& fit) {
  int64_t longest = 0, total = 0;
  for (int r = 0; r < n_req; ++r) {
    longest = std::max(longest, tiles[r]);
    total += tiles[r] * Hkv;
  }
  const int64_t pairs = (int64_t)n_req * Hkv;
  DecodePlan p = {1, 0};
  for (int k = 1; k < kClusterKinds && (int64_t)p.cluster * kDecTileWarps < longest; ++k)
    if (fit.n[k] >= pairs) p.cluster = kClusterSizes[k];
  const double slots = std::max(1, fit.n[0]);
  const double even = (double)total / (slots * kDecTileWarps);
  const double mean = (double)total / ((double)pairs * p.cluster * kDecTileWarps);
  const double last = (double)longest / (p.cluster * kDecTileWarps);
  // pairs that do not fit at once run in waves of mean length; the longest may end last
  const int64_t waves = p.cluster > 1 ? 1 : (pairs + (int64_t)slots - 1) / (int64_t)slots;
  if ((double)waves * mean + (last - mean) > kEvenCost * even + kPartCost) {
    const int64_t spread = std::min<int64_t>(kPartMax, std::max<int64_t>(kPartMin, (int64_t)even + 1));
    const int64_t fewest = (longest + kPartsMax * kDecTileWarps - 1) / (kPartsMax * kDecTileWarps);
    p.cluster = 1;
    p.part_tiles = kDecTileWarps * (int)std::max(spread, fewest);
  }
  return p;
}

}  // namespace vc
