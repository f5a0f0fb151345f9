// Geometry and launch parameters of the register-tile kernel (tiles.cuh).
#pragma once

#include <cuda_runtime.h>

#include "runtime.h"

namespace sdfg {

constexpr int TK_DOWN = 20;                       // binary orders a tile with large values is scaled down by
constexpr int TK_HALO = 8;                        // halo rows and columns = steps per pass
constexpr int TK_W = 128;                         // box columns, 4 per lane
constexpr int TK_TX = TK_W - 2 * TK_HALO;         // 112 columns per tile

struct TileParams {
    const void *in;
    void *out;
    uint64_t *xrows;  // exchange words (zero before the launch), for two passes each:
    uint64_t *xcols;  // [2][ny][2][8][ldx] and [2][nx][2][R][8]
    int *err;         // device error word
    int R, C, ld, ldx;
    int nx, ny;       // tiles
    int vec;          // rows can be read and written four columns at a time
    int n_pass, k_last;  // passes, steps (SOR: half-sweeps) of the last one
    // the factor at the end of a pass as hi + lo: 0.2^8 and 0.2^k_last, and the
    // same times 2^TK_DOWN for tiles with large values
    struct Factor {
        float hi, lo;
    } factor[2], factor_large[2];
    float a, b;       // SOR: 1 - omega, omega / 4
    unsigned long long timeout_ns;
    unsigned stuck;  // test hook: the halo waits are for passes that far ahead (0: none)
};

// First column and row of a tile: the first tile starts at 0, the last ends at
// (columns: within 3 of) the grid's end, the others lie evenly between, columns
// at multiples of 4.  (A grid has at most some thousand tiles: no overflow.)
__host__ __device__ inline int tile_x0_of(int C, int nx, int tx) {
    return nx > 1 ? tx * ((C - TK_TX + 3) / 4) / (nx - 1) * 4 : 0;
}
__host__ __device__ inline int tile_y0_of(int R, int ny, int ty, int TY) {
    return ny > 1 ? ty * (R - TY) / (ny - 1) : 0;
}
__host__ __device__ inline int tile_x0(const TileParams &p, int tx) { return tile_x0_of(p.C, p.nx, tx); }
__host__ __device__ inline int tile_y0(const TileParams &p, int ty, int TY) { return tile_y0_of(p.R, p.ny, ty, TY); }

// A variant of the kernel: nw warps per CTA, each holding rb rows.
struct TileShape {
    int nw, rb;
};
struct TilePlan {
    TileShape shape;
    int nx, ny;
};
inline int tile_rows(TileShape v) { return v.nw * v.rb - 2 * TK_HALO; }  // rows a tile answers for
inline size_t tile_smem(TileShape v) { return sizeof(float) * v.nw * v.rb * TK_W; }

}  // namespace sdfg
