// Tiling of the 3D z-march kernels (lks_march3d.cu, lks_march3d_adj.cu).
#pragma once

#include "lks_internal.h"

namespace lks {

// What a kernel's tiles look like and what its blocks cost.
struct MarchCost {
    int tile_x;               // output columns of a tile
    int rows, halo;           // a block of w warps covers rows w - halo output rows
    int max_warps, room;      // per block, resident per SM
    double wave, tail;        // a plane of a wave of k resident warps per SM: wave + k; tail: the
                              // blocks at the faces, which finish last
    double start;             // planes a block pays for its halo, besides 8 / (blocks per SM) to
                              // fill its ring while the SM's other blocks run
};

// Tiles over out_x columns, out_y rows and chunks of nz planes: the block height (4 warps or more;
// warps > 0 fixes it) and the chunk (8 planes or more) with the least cost.  The constants of
// MarchCost are fits to the times of 80 tilings of 256^3, 128^3, 151 x 83 x 117 and 96 x 90 x 101
// for each kernel (residual 3 % for the forward step, 5 % for the adjoint; the tilings of one grid
// differ by up to a third).  On 60 other grids the forward cost predicts the step's time within 6 %.
March3d march_tiles(const MarchCost& m, int out_x, int out_y, int nz, int warps);

// Tiles of the forward march, and the interior nodes of one forward step on them.
March3d step_march_tiles(const Geom& g);
cudaError_t launch_step_march(const Geom& g, const V4<float>* src, const V4<float>* kus,
                              V4<float>* dst, int* err, cudaStream_t st, const March3d& t);
// Tiles of the adjoint march in blocks of `warps` warps (0: by cost), the first of 32 columns from column
// org, -2 or 0, the next 28 on.  A tile's first and last two columns are halo, but with org 0 those at the
// faces: a grid of 28 t + 4 columns then takes t tiles, and 28 t with org -2.
constexpr int kAdjTileX = 28;
March3d adj_march_tiles(const Geom& g, int org, int warps);
// lambda^{n-1} from lambda^n (after k_adj_prep) but for the one-sided boundary rows, whose 2 A S~ go
// to face.
cudaError_t launch_adj_march(const Geom& g, const V4<float>* lam_in, V4<float>* lam_out,
                             const V4<float>* sp, float* face, int* err, cudaStream_t st,
                             const March3d& t, int org);

}  // namespace lks
