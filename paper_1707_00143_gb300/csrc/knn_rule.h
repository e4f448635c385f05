// knn_rule.h -- which of the two tensor-core kNN kernels a call runs: host
// arithmetic only.
#pragma once

#include <algorithm>
#include <cstdint>

namespace nsg {

// Base tiles (128 rows) that the pre-pass of knn_tc.cu samples to bound the
// rank-th distance, 0: too few for a useful bound.  Two minima per tile, 2.5
// ranks' worth of tiles: the bound then admits ~1.1 times the sample's own k
// nearest, and a larger sample would cost more tiles than the candidates it
// saves (k ln 2 per doubling, ~30 warp instructions each, against ~10 per tile
// and row).  At most a quarter of the base.
inline int knn_sample_tiles(int64_t ntiles, int rank) {
    const int p = (int)std::min<int64_t>(ntiles / 4, (int64_t)rank * 5 / 2);
    return 2 * p >= rank + rank / 4 ? p : 0;
}

// Whether a call runs the kernel whose scanning warps merge themselves, a CTA
// per 128 query rows (knn_tc_small.cu), instead of the one of 256-row units with
// separate merging warps, splits and pre-pass (knn_tc.cu).  KL: entries per list;
// bounded: the pre-pass has enough tiles.
//
// Bounded, the units' scan is the faster one and their pre-pass, rings and
// launches are what short bases do not pay back: 200 us more for one query,
// and for many queries on few rows (12,000 x 128, KL = 10: 8,000 queries
// 1.04 times the units' speed, 1,500 0.73).  Rows in tight clusters side by side
// get little from the pre-pass (20,000-row graph, K = 10, clusters of 100: 2,604 us,
// units 4,156; 60,000 rows: equal).  Unbounded, nearly every
// column is a candidate and merging is the work: a unit's wave takes ~1.8 times
// a CTA wave (40,000 x 96, KL = 150, 10,000 queries: 4,845 us, units 6,763), so
// units win when they finish in one wave where the CTAs need two (26,000-row
// graph, K = 100: 5,340 us, units 4,319; fewer than 2/3 of the SMs' worth of units are
// split, which lengthens the merging: 24,000 queries, KL = 200, 9,742 us, units
// 15,484), or few queries leave the CTAs' SMs idle (26,000 x 96, KL = 150, 300
// queries: 3,861 us, units 2,788; 12,000 x 96, KL = 42: 1,403 and 1,544).
inline bool knn_small(int64_t n, int64_t nq, int KL, bool bounded, int sms) {
    const int64_t ctas = (nq + 127) / 128, units = (nq + 255) / 256;
    const bool one_wave = ctas > sms && units <= sms;
    if (bounded) return !(n >= 20480 || (n >= (nq < 32 ? 16384 : 8192) && 3 * nq <= n && nq <= 2048));
    return !(KL >= 64 && ((n >= 10240 && nq <= 2048) || (n >= 20000 && one_wave && 3 * units > 2 * sms)));
}

}  // namespace nsg
