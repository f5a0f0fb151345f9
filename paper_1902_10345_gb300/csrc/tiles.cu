// Planning and launch of the register-tile kernel (tiles.cuh).
#include <math.h>
#include <string.h>

#include <algorithm>

#include "launchset.h"
#include "per_device.h"
#include "tiles.cuh"

namespace sdfg {

const void *tile_fn_mid(int rb, int dtype);   // tiles_mid.cu: 16 warps, up to 9 rows
const void *tile_fn_tall(int rb, int dtype);  // tiles_tall.cu: up to 12
const void *tile_fn_top(int rb, int dtype);   // tiles_top.cu: up to 18
const void *sor_tile_fn(TileShape v, int dtype);       // sor_tiles.cu
const void *sor_tile_fn_tall(TileShape v, int dtype);  // sor_tiles_tall.cu: 16 warps, 10 rows and more

namespace {
constexpr TileShape kShapes[] = {{8, 4},   {8, 5},   {8, 6},   {8, 7},   {16, 4},  {16, 5},  {16, 6},  {16, 7}, {16, 8},
                                 {16, 9},  {16, 10}, {16, 11}, {16, 12}, {16, 14}, {16, 16}, {16, 17}, {16, 18}};
constexpr int kShapeCount = sizeof(kShapes) / sizeof(kShapes[0]);
bool sor_has(TileShape v) { return v.nw == 8 ? v.rb % 2 == 0 : v.rb % 2 == 0 ? v.rb < 16 : v.rb == 17; }

const void *tile_fn(TileShape v, int dtype, bool sor) {
    if (sor) return v.nw == 16 && v.rb >= 10 ? sor_tile_fn_tall(v, dtype) : sor_tile_fn(v, dtype);
    if (v.nw == 16) return v.rb <= 9 ? tile_fn_mid(v.rb, dtype) : v.rb <= 12 ? tile_fn_tall(v.rb, dtype) : tile_fn_top(v.rb, dtype);
    switch (v.rb) {
        case 4: return tile_fn_of<8, 4>(dtype);
        case 5: return tile_fn_of<8, 5>(dtype);
        case 6: return tile_fn_of<8, 6>(dtype);
        default: return tile_fn_of<8, 7>(dtype);
    }
}

// CTAs of variant `i` an SM holds (a property of the compiled kernel), and the
// kernel's shared-memory limit raised: both on the current device, which is `device`
int tile_blocks_per_sm(int i, int dtype, bool sor, int device) {
    static PerDevice<kShapeCount * 4> known;
    return known.get(device, (i * 2 + (dtype == SDFG_BF16)) * 2 + sor, [&]() {
        const TileShape v = kShapes[i];
        const void *fn = tile_fn(v, dtype, sor);
        int n = 0;
        if (cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(tile_smem(v))) != cudaSuccess ||
            cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, fn, 32 * v.nw, tile_smem(v)) != cudaSuccess) {
            cudaGetLastError();
            return 0;
        }
        return n;
    });
}

// Tiles along an axis of n points when a tile answers for t of them.
int tiles_along(int n, int t) { return n <= t ? 1 : (n + t - 1) / t; }

// Whether the halo of every tile but those at the grid's ends lies in its two
// neighbours, and holds a point of the boundary ring in its outermost row or
// column at most (which is wrong after one step in any case).  `apart`: what lies
// between two tiles with one in between (the halo; along columns twice that,
// so that no lane holds halo columns of both neighbours).
template <class First> bool halos_in_neighbours(int n, int extent, int tile, int apart, First first) {
    if (n == 1) return true;
    if (first(1) < TK_HALO || first(n - 2) + tile + TK_HALO > extent) return false;
    for (int i = 0; i + 2 < n; ++i)
        if (first(i + 2) - first(i + 1) < TK_HALO || first(i + 2) < first(i) + tile + apart) return false;
    return true;
}
}  // namespace

// The variant and tile counts for a grid, or false when none holds it.  The
// time of a pass is estimated as 8 steps of the warps a scheduler has: 14 pipe
// cycles a row, and some hundred a step for the barrier, the shuffles and the
// neighbouring band's row.  Measured best and chosen: 256^2 T=100 8 warps x 4
// rows (50 us; 7 rows 54, 16 x 4 60), 1301 x 1777 T=150 16 x 12 (146 us) and
// 16 x 11 (148), 2048^2 T=1024 16 x 17 (1345 us; 16 x 18 1450).
bool plan_tiles(int R, int C, int dtype, const DeviceState *st, TilePlan *plan, bool sor) {
    const int sm_count = st->sm_count;
    if (dtype == SDFG_F64 || R < 3 || C < 3) return false;
    const int x = tiles_along(C, TK_TX);
    if (x > 4LL * sm_count) return false;
    if (!halos_in_neighbours(x, C, TK_TX, 2 * TK_HALO, [&](int t) { return tile_x0_of(C, x, t); })) return false;
    double best = 0.0;
    for (int i = 0; i < kShapeCount; ++i) {
        const TileShape v = kShapes[i];
        if (sor && !sor_has(v)) continue;
        const int TY = tile_rows(v);
        if (R < TY) continue;  // the ring rows lie at fixed box rows: a tile is no taller than the grid
        const int y = tiles_along(R, TY);
        const long long n = static_cast<long long>(x) * y;
        if (n > 4LL * sm_count) continue;
        const int per_sm = static_cast<int>((n + sm_count - 1) / sm_count);
        const double cost = 8.0 * (14.0 * v.rb * (v.nw / 4) * per_sm + 250.0);
        // (the cost first: walking the tiles of every shape took a third of a short
        // call on a grid of many, 3000 x 48 T=1 15.2 us)
        if (best != 0.0 && cost >= best) continue;
        if (n <= static_cast<long long>(tile_blocks_per_sm(i, dtype, sor, st->device)) * sm_count &&
            halos_in_neighbours(y, R, TY, TK_HALO, [&](int t) { return tile_y0_of(R, y, t, TY); })) {
            best = cost;
            plan->shape = v;
            plan->nx = x;
            plan->ny = y;
        }
    }
    return best > 0.0;
}

int run_tiles(const void *in, void *out, int R, int C, int ld, long long T, int dtype, const TilePlan &plan,
              DeviceState *st, cudaStream_t s, const double *omega) {
    const int nx = plan.nx, ny = plan.ny;
    TileParams p;
    memset(&p, 0, sizeof(p));
    p.in = in;
    p.out = out;
    p.err = st->d_err;
    p.R = R;
    p.C = C;
    p.ld = ld;
    p.ldx = (C + 31) / 32 * 32;
    p.nx = nx;
    p.ny = ny;
    const size_t quad = 4 * static_cast<size_t>(dtype_bytes(dtype));
    p.vec = reinterpret_cast<uintptr_t>(in) % quad == 0 && reinterpret_cast<uintptr_t>(out) % quad == 0 && ld % 4 == 0;
    const int per_step = omega ? 2 : 1;  // an SOR iteration is two half-sweeps, each a cell of halo
    p.n_pass = static_cast<int>((T * per_step + TK_HALO - 1) / TK_HALO);
    p.k_last = static_cast<int>(T * per_step - static_cast<long long>(p.n_pass - 1) * TK_HALO);
    if (omega) {
        p.a = static_cast<float>(1.0 - *omega);
        p.b = static_cast<float>(0.25 * *omega);
    }
    for (int last = 0; last < 2; ++last) {
        double f = 1.0;
        for (int i = 0; i < (last ? p.k_last : TK_HALO); ++i) f = 0.2 * f;
        auto split = [](double v, bool down) {
            TileParams::Factor q;
            q.hi = static_cast<float>(v);
            // (rounded down the low half is positive: an infinity keeps its sign)
            if (down && q.hi > v) q.hi = nextafterf(q.hi, 0.0f);
            q.lo = static_cast<float>(v - static_cast<double>(q.hi));
            return q;
        };
        p.factor[last] = split(f, false);
        p.factor_large[last] = split(ldexp(f, TK_DOWN), true);
    }
    p.timeout_ns = test_hooks().timeout_ns ? test_hooks().timeout_ns : DEFAULT_TIMEOUT_NS;
    p.stuck = test_hooks().inject_stuck_wait ? LL_NEVER : 0;
    // exchange words for two passes, and where a single pass works in place,
    // a grid for the result: a tile may not store what a neighbour still has to load
    const bool staged = in == out && p.n_pass == 1;
    const size_t n_rows = static_cast<size_t>(4 * TK_HALO) * ny * p.ldx, n_cols = static_cast<size_t>(4 * TK_HALO) * nx * R;
    const size_t words = p.n_pass > 1 ? (n_rows + n_cols) * sizeof(uint64_t) : 0;
    const size_t bytes = staged ? static_cast<size_t>(R) * ld * dtype_bytes(dtype) : words;
    void *ws = nullptr;
    int rc = scratch_alloc(&ws, bytes, s);
    if (rc != SDFG_OK) return rc;
    p.xrows = static_cast<uint64_t *>(ws);
    p.xcols = p.xrows + n_rows;
    if (staged) p.out = ws;
    cudaError_t e = words ? cudaMemsetAsync(ws, 0, words, s) : cudaSuccess;
    if (e == cudaSuccess) {
        void *args[] = {&p};
        TimedLaunch t = stats_begin(omega ? FAM_SOR : FAM_RESIDENT, s);
        e = cudaLaunchCooperativeKernel(tile_fn(plan.shape, dtype, omega != nullptr), dim3(nx * ny), dim3(32 * plan.shape.nw), args,
                                        tile_smem(plan.shape), s);
        stats_end(t, s);
    }
    if (e == cudaErrorCooperativeLaunchTooLarge) {
        cudaGetLastError();  // the tiles do not fit side by side (a partition of the device): the caller's other path
        rc = SDFG_ERR_NOMEM;
    } else if (e != cudaSuccess) {
        rc = cuda_error(e, "register-tile launch");
    }
    if (rc == SDFG_OK && staged) rc = launch_copy2d(out, ld, ws, ld, R, C, dtype, s);
    scratch_free(ws, s);
    return rc;
}

}  // namespace sdfg
