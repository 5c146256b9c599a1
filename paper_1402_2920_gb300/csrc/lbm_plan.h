// Rules that choose kernels and launch shapes from a lattice's size.  Plain host functions.
#pragma once

#include <cstdint>

namespace lbm {

// rows of CTAs that a grid can have
constexpr int64_t kGridRows = 65535;
// sites of a tile of the pairwise collision: 64 x 4 or 32 x 8
constexpr int kPairTileSites = 256;
constexpr int pair_tile_rows(int width) { return kPairTileSites / width; }

// whether x-neighbouring sites (2k, 2k + 1) are aligned words of every field plane
inline bool pairs_of_sites(const int64_t dims[3]) { return dims[0] % 2 == 0; }

// Whether the pairwise collision takes tiles of 64 x 4 sites (else 32 x 8): where they pad nx by at most a
// fifth more, and the grid has the rows.  Measured, 64 / 32 wide: 256^3 1.17 / 1.59 ms, 192^3 0.49 / 0.56, 128^3
// 0.150 / 0.160; padded by a fifth, 160^3 0.330 / 0.369, 144^3 0.264 / 0.270, 132 x 256 x 256 0.83 / 0.89,
// 130 x 128 x 128 0.226 / 0.216; by a third, 96^3 0.087 / 0.076; 48^3 14 / 15 us.
inline bool wide_tiles(const int64_t dims[3])
{
    const int64_t w32 = (dims[0] + 31) / 32 * 32, w64 = (dims[0] + 63) / 64 * 64;
    return 5 * w64 <= 6 * w32 && dims[1] <= kGridRows * pair_tile_rows(64);
}

}  // namespace lbm
