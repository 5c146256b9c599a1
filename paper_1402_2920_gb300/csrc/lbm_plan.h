// Rules that choose kernels and launch shapes from a lattice's size.  Plain host functions.
#pragma once

#include <cstdint>

#include "lbm.h"

namespace lbm {

// rows of CTAs that a grid can have
constexpr int64_t kGridRows = 65535;
// sites of a tile of the pairwise collision: 64 x 4 or 32 x 8
constexpr int kPairTileSites = 256;
constexpr int pair_tile_rows(int width) { return kPairTileSites / width; }

// whether x-neighbouring sites (2k, 2k + 1) are aligned words of every field plane
inline bool pairs_of_sites(const int64_t dims[3]) { return dims[0] % 2 == 0; }

// Whether the pairwise collision takes tiles of 64 x 4 sites (else 32 x 8): where they pad nx by at most a
// fifth more, and the grid has the rows.  Measured, 64 / 32 wide: 256^3 1.17 / 1.59 ms, 192^3 0.50 / 0.56, 160^3 (padded
// by a fifth) 0.333 / 0.329, 128^3 0.155 / 0.160, 96^3 (a third) 0.087 / 0.076, 48^3 14 / 15 us.
inline bool wide_tiles(const int64_t dims[3])
{
    const int64_t w32 = (dims[0] + 31) / 32 * 32, w64 = (dims[0] + 63) / 64 * 64;
    return 5 * w64 <= 6 * w32 && dims[1] <= kGridRows * pair_tile_rows(64);
}

// Whether the sweeps are in FP64.
inline bool usolve_f64(const lbm_params& prm)
{
    return prm.storage == LBM_STORE_F64 || prm.usolve_precision == LBM_USOLVE_F64;
}

// Derivatives and collision on pairs of sites: 0 not, 1 with tiles 32 wide, 2 with tiles 64 wide.  They exist in 3D
// for FP32 deviations with FP32 sweeps (KernelTable::pair_derivs) and need aligned pairs.
inline int pair_class(int lattice, const int64_t dims[3], const lbm_params& prm)
{
    if (lattice != LBM_D3Q59 || prm.storage != LBM_STORE_F32_DEV || usolve_f64(prm) || !pairs_of_sites(dims)) return 0;
    return wide_tiles(dims) ? 2 : 1;
}

// Batch key of a simulation: its kernels and its size class (sites within a factor of 4).  Simulations batch
// together only when their keys are equal: a batch runs one set of kernels and steps in lockstep, so a small
// simulation beside a much larger one would wait for it at every stage.
inline int batch_key(int lattice, const int64_t dims[3], const lbm_params& prm)
{
    const int kernels = (((lattice * 16 + prm.storage) * 2 + (usolve_f64(prm) ? 1 : 0)) * 2 + (prm.gamma != 0.0 ? 1 : 0)) * 3 +
                        pair_class(lattice, dims, prm);
    int64_t n = dims[0] * dims[1] * (lattice == LBM_D3Q59 ? dims[2] : 1);
    int size_class = 0;
    while (n >= 4) {
        n >>= 2;
        ++size_class;
    }
    return kernels * 64 + size_class;
}

}  // namespace lbm
