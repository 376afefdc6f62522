// matmul_tile.h -- the tile width of the tensor matmul (host code only).
#pragma once

#include <cstdint>

namespace ccm {
namespace tc {

constexpr int kBM = 256;  // rows of C per CTA pair (128 per CTA)

// The instances: 32-bit accumulators, and 64-bit ones.
constexpr int kTileCols32[] = {256, 224, 192, 128, 64}, kTileCols64[] = {128, 64};

// Columns of a tile of an m x n product on `pairs` CTA pairs: the width with the
// least loading.  The L2 feeds about 46 bytes per clock and SM (256 columns: 32 KB
// per block of k, 90 us at 4096^3; 128: 24 KB, 111 us), so a wave of tiles costs
// 128 rows of A and half a tile width of B per CTA whatever the MMAs cost.  At
// 4096^3: 224 columns give exactly 4 waves, 82 us.
inline int tile_columns(uint64_t m, uint64_t n, bool acc32, uint64_t pairs) {
  const int* cols = acc32 ? kTileCols32 : kTileCols64;
  const int count = acc32 ? 5 : 2;
  const uint64_t tiles_m = (m + kBM - 1) / kBM;
  int chosen = 0;
  double least = 0;
  for (int i = 0; i < count; ++i) {
    const uint64_t tiles = tiles_m * ((n + cols[i] - 1) / cols[i]);
    const uint64_t waves = (tiles + pairs - 1) / pairs;
    const double cost = (double)waves * (256 + cols[i]);
    if (!chosen || cost < least) {
      chosen = cols[i];
      least = cost;
    }
  }
  return chosen;
}

}  // namespace tc
}  // namespace ccm
