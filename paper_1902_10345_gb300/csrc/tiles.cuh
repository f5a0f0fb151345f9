// Register tiles: every step of one FP32/BF16 grid in ONE cooperative launch,
// the grid held in registers from the first step to the last (StateFusion over
// the whole state loop, paper App. B; the array itself is the LocalStorage).
//
// A CTA of NW warps owns a box of NW RB rows x 128 columns: the tile it is
// responsible for, TY = NW RB - 16 rows x 112 columns, and a halo of 8 on each
// side.  Each warp holds RB consecutive box rows in registers, 4 columns per
// lane, and advances them in place, 8 steps per pass; values that are wrong
// for want of a neighbour outside the box spread one row and one column per
// step, so the halo absorbs a pass.  Between passes the box goes through
// shared memory: a tile writes the rows and columns that its neighbours hold
// as halo to a global exchange buffer and reads its own halo from it, so no
// HBM traffic happens between the first load and the final store.
//
// The exchange words carry the number of their pass (ll_store, ll_load): no
// fence, no flag, no grid barrier.  Two buffers alternate; a tile overwrites
// what it wrote two passes ago only after it has read the last pass's words of
// every neighbour, which each neighbour wrote after reading those of the pass
// before.  Measured on 256^2 (48 tiles): 4.0 us per pass with release/acquire
// flags per tile, of which 4/5 exchange, 2.9 us with stamped words.
//
// What bounds it: issue of the steps (2048^2, 16 warps x 17 rows, 152 tiles,
// one per SM: 14100 of 21900 cycles per pass; a row is 6 FADD + 4 FADD2 + 2
// SHFL and about 4 moves for 4 points per lane, 14 pipe cycles), then the
// exchange (about 3300 cycles), then the box's way through shared memory.
// Bigger tiles recompute less halo (1.21x at 16 x 17), which counts for more
// than a second CTA per SM would hide: all tiles wait for each other every
// pass, so two CTAs of an SM compute at the same time and wait at the same
// time (12.4 us per pass with 304 tiles of 8 x 18, 10.9 with 152).
//
// The same kernel runs red-black SOR (SOR: 8 half-sweeps, 4 iterations, per
// pass, in the exact order of sor2d.cu).
//
// Arithmetic (Jacobi): (n + (w + c + e)) + s with shared pair sums, unscaled (after t
// steps of a pass the tile holds 5^t times the state), one multiplication by
// 0.2^8 (hi + lo) at the end of a pass.  The order does not depend on a
// point's place in its tile, so the tiling changes no bit.  The boundary ring
// is multiplied by 5 each step (as every value is, in effect) and set back to
// its exact value at the end of a pass.  Points outside the grid may take any
// value: they reach the interior only through the ring.  BF16 grids stay FP32
// from load to store.  A tile that has loaded or received a value of SCALED_LIMIT or
// more computes 2^-20 of it from then on (a power of two, which changes no
// bit of what is not as small as 2^-106), so that no sum overflows which would
// not in the plain order; no other tile can get one, as a step averages.
// (The test of what each exchange brings and of the flag is some 20 instructions a
// pass, which cost nothing measurable on the tallest tiles, 2048^2 T=1024 1348 -> 1331 us,
// and up to 5% of FP32 and 9% of BF16 passes on grids of 400^2 to 1000^2, 1000^2 T=300 180 ->
// 189 and 176 -> 188 us.  A kernel in the memset's place that looks the grid over first
// spares those and costs the tall ones 4%; an agreement between the tiles during the
// first pass cost as much as the test.)
#pragma once

#include <type_traits>

#include "exchange.cuh"
#include "sor_row.cuh"
#include "tiles.h"

namespace sdfg {

template <int I, int N, class F> __device__ __forceinline__ void tk_for(F &&f) {
    if constexpr (I < N) {
        f(std::integral_constant<int, I>());
        tk_for<I + 1, N>(f);
    }
}

// The horizontal three-point sums (w + c + e) of a lane's four columns, with
// shared pair sums.
__device__ __forceinline__ void tk_h3(float (&h)[4], const float (&x)[4]) {
    const float left = __shfl_up_sync(FULL_MASK, x[3], 1);
    const float right = __shfl_down_sync(FULL_MASK, x[0], 1);
    const float q0 = __fadd_rn(x[0], x[1]);
    const float q1 = __fadd_rn(x[2], x[3]);
    h[0] = __fadd_rn(left, q0);
    h[1] = __fadd_rn(q0, x[2]);
    h[2] = __fadd_rn(x[1], q1);
    h[3] = __fadd_rn(q1, right);
}
// Two columns per packed add.  (Pairs as a 16-byte access leaves them: pairing
// columns 0, 2 and 1, 3 packs one add more per row, but then the compiler moves
// 16 registers a row to form the pairs; 17.6 against 13.4 us per 2048^2 pass.)
__device__ __forceinline__ void tk_add(float (&o)[4], const float (&a)[4], const float (&b)[4]) {
#pragma unroll
    for (int e = 0; e < 4; e += 2) {
        const float2 t = __fadd2_rn(make_float2(a[e], a[e + 1]), make_float2(b[e], b[e + 1]));
        o[e] = t.x;
        o[e + 1] = t.y;
    }
}
__device__ __forceinline__ void tk_copy(float (&o)[4], const float (&a)[4]) {
#pragma unroll
    for (int e = 0; e < 4; ++e) o[e] = a[e];
}

// Where a tile lies and what it shares with its neighbours; computed once by
// one thread (a dozen divisions) and kept in shared memory, where each phase
// reads it anew: held across the steps it would cost the registers that the
// band needs.
struct TilePlace {
    int tx, ty;
    int x0, y0, x1, y1;  // the tile answers for rows [y0, y1), columns [x0, x1): up to the next tile's first
    // what the neighbours hold as halo: 8 rows from rn for the tiles above, 8
    // from rs for those below, 8 columns from cw for those to the west and 8
    // from ce for those to the east (far off the tile where there is none)
    int rn, rs, cw, ce;
    __device__ __forceinline__ void set(const TileParams &P, int TY) {
        constexpr int NONE = -(1 << 30);
        tx = blockIdx.x % P.nx;
        ty = blockIdx.x / P.nx;
        x0 = tile_x0(P, tx);
        y0 = tile_y0(P, ty, TY);
        x1 = tx + 1 < P.nx ? tile_x0(P, tx + 1) : P.C;
        y1 = ty + 1 < P.ny ? tile_y0(P, ty + 1, TY) : P.R;
        rn = ty > 0 ? tile_y0(P, ty - 1, TY) + TY : NONE;
        rs = ty + 1 < P.ny ? y1 - TK_HALO : NONE;
        cw = tx > 0 ? tile_x0(P, tx - 1) + TK_TX : NONE;
        ce = tx + 1 < P.nx ? x1 - TK_HALO : NONE;
    }
};

template <class ST, int NW, int RB, bool SOR>
__global__ void __launch_bounds__(32 * NW, 16 / NW) tile_kernel(const __grid_constant__ TileParams P) {
    constexpr int NT = 32 * NW;
    constexpr int BY = NW * RB;
    constexpr int TY = BY - 2 * TK_HALO;
    static_assert(RB >= 4 && TY >= 16, "a tile is at least two halos high");
    // the box between two passes (and on its way from and to the grid): the
    // registers hold it during a pass
    extern __shared__ __align__(16) float box_smem[];
    float(*const box)[TK_W] = reinterpret_cast<float(*)[TK_W]>(box_smem);
    // band-edge rows, double-buffered by step parity: top[p][w] is warp w's
    // first row, bot[p][w + 1] its last; bot[p][0] and top[p][NW] stand for
    // the rows beyond the box (zeros)
    __shared__ __align__(16) float4 top[2][NW + 1][32];
    __shared__ __align__(16) float4 bot[2][NW + 1][32];
    __shared__ float ring_col[2][BY];      // exact values of columns 0 and C-1 in this box's rows
    __shared__ float ring_row[2][TK_W];    // and of rows 0 and R-1 in its columns
    __shared__ TilePlace place;
    __shared__ int large;  // the box holds, or has held, a value of SCALED_LIMIT or more (Jacobi)

    const int R = P.R, C = P.C;
    const int tid = threadIdx.x;
    const int lane = tid & 31;
    const int warp = tid >> 5;
    if (tid == 0) {
        place.set(P, TY);
        large = 0;
    }
    __syncthreads();
    // (an opaque pointer: see TilePlace)
    auto where = [&]() {
        const TilePlace *p = &place;
        asm volatile("" : "+l"(p));
        return p;
    };

    float X[RB][4];  // the band's rows
    auto put = [&](float4 *slot, const float(&x)[4]) { slot[lane] = make_float4(x[0], x[1], x[2], x[3]); };
    auto get = [&](float(&x)[4], const float4 *slot) {
        const float4 v = slot[lane];
        x[0] = v.x;
        x[1] = v.y;
        x[2] = v.z;
        x[3] = v.w;
    };
    float4 *const band = reinterpret_cast<float4 *>(box[warp * RB]);  // the band's rows, 32 float4 each
    auto take_band = [&]() {
        tk_for<0, RB>([&](auto i_t) {
            constexpr int i = decltype(i_t)::value;
            get(X[i], band + i * 32);
        });
        if constexpr (!SOR) {
            if (large) {
                constexpr float DOWN = 1.0f / (1 << TK_DOWN);
                tk_for<0, RB>([&](auto i_t) {
#pragma unroll
                    for (int e = 0; e < 4; ++e) X[decltype(i_t)::value][e] *= DOWN;
                });
            }
        }
    };
    // (every thread that finds one writes the same; read after the next barrier)
    auto note_large = [&](float m) {
        if (!SOR && m >= SCALED_LIMIT) large = 1;
    };

    // The boundary ring in this box.  Tile row 0 starts at grid row 0 and the
    // last tile row ends at row R-1, so the ring rows are box rows HALO and
    // BY - HALO - 1 at compile time; column 0 is box column HALO, column C-1
    // box column `rq` of the last tile column, element `er` of its lane.
    constexpr int WT = TK_HALO / RB, IT = TK_HALO % RB;
    constexpr int WB = (BY - TK_HALO - 1) / RB, IB = (BY - TK_HALO - 1) % RB;
    int rq, er, variant;  // variant: which ring columns the box holds (see step)
    bool lane_l, lane_r, fix_top, fix_bot;
    {
        const TilePlace g = *where();
        const int gx = g.x0 - TK_HALO + lane * 4;   // grid column of the lane's element 0
        const int yb = g.y0 - TK_HALO + warp * RB;  // grid row of the band's first row
        const bool quad_in = gx >= 0 && gx + 4 <= C && P.vec;
        const ST *p = static_cast<const ST *>(P.in) + static_cast<ptrdiff_t>(yb) * P.ld + gx;
        float m = 0.f;  // (fmaxf passes a NaN over)
#pragma unroll 6
        for (int i = 0; i < RB; ++i, p += P.ld) {
            float v[4] = {0.f, 0.f, 0.f, 0.f};
            if (yb + i >= 0 && yb + i < R) {
                if (quad_in) {
                    VecIO<ST, 4>::load(v, p);
                } else {
#pragma unroll
                    for (int e = 0; e < 4; ++e)
                        if (gx + e >= 0 && gx + e < C) v[e] = to_ct<ST>(p[e]);
                }
            }
            put(band + i * 32, v);
#pragma unroll
            for (int e = 0; e < 4; ++e) m = fmaxf(m, fabsf(v[e]));
        }
        note_large(m);
        const bool has_l = g.tx == 0, has_r = g.tx == P.nx - 1;
        rq = C - 1 - (g.x0 - TK_HALO);
        er = rq & 3;
        lane_l = has_l && lane == TK_HALO / 4;
        lane_r = has_r && lane == (rq >> 2);
        fix_top = g.ty == 0 && warp == WT;
        fix_bot = g.ty == P.ny - 1 && warp == WB;
        variant = has_l ? (has_r ? 6 : 1) : has_r ? 2 + er : 0;
        __syncthreads();
        take_band();
        if (tid < BY && has_l) ring_col[0][tid] = box[tid][TK_HALO];
        if (tid < BY && has_r) ring_col[1][tid] = box[tid][rq];
        if (tid < TK_W) ring_row[0][tid] = box[TK_HALO][tid];
        if (tid < TK_W) ring_row[1][tid] = box[BY - TK_HALO - 1][tid];
    }
    if (warp == 0) {
        const float4 z = make_float4(0.f, 0.f, 0.f, 0.f);
        bot[0][0][lane] = bot[1][0][lane] = z;
        top[0][NW][lane] = top[1][NW][lane] = z;
    }

    // One step.  The bands' edge rows of this step's start are in slot p; the
    // rows that need no other band's row come first, so the barrier and the
    // reads of the neighbours' rows overlap them.  CF: 0 no ring column, 1
    // column 0, 2 + e column C-1 at element e, 6 both.
    auto step = [&](auto cf_t, int slot) {
        constexpr int CF = decltype(cf_t)::value;
        auto fix = [&](auto i_t, float(&o)[4], const float(&c)[4]) {
            constexpr int i = decltype(i_t)::value;
            if constexpr (CF == 1 || CF == 6) {
                if (lane_l) o[0] = __fmul_rn(5.0f, c[0]);
            }
            if constexpr (CF >= 2 && CF <= 5) {
                if (lane_r) o[CF - 2] = __fmul_rn(5.0f, c[CF - 2]);
            }
            if constexpr (CF == 6) {
#pragma unroll
                for (int e = 0; e < 4; ++e)
                    if (lane_r && er == e) o[e] = __fmul_rn(5.0f, c[e]);
            }
            if constexpr (i == IT || i == IB) {
                if ((i == IT && fix_top) || (i == IB && fix_bot)) {
#pragma unroll
                    for (int e = 0; e < 4; ++e) o[e] = __fmul_rn(5.0f, c[e]);
                }
            }
        };
        float x1[4];     // old row 1: row 0's south
        float xz[4];     // old row RB-2: the last row's north
        float p[4];      // north + (w + c + e) of the row being updated
        tk_copy(x1, X[1]);
        {
            float h[4];
            tk_h3(h, X[1]);
            tk_add(p, X[0], h);
        }
        tk_for<1, RB - 1>([&](auto i_t) {
            constexpr int i = decltype(i_t)::value;
            float pn[4], o[4];
            if constexpr (i + 1 < RB - 1) {
                float h[4];
                tk_h3(h, X[i + 1]);
                tk_add(pn, X[i], h);
            } else {
                tk_copy(xz, X[i]);
                tk_copy(pn, p);
            }
            tk_add(o, p, X[i + 1]);
            fix(i_t, o, X[i]);
            tk_copy(X[i], o);
            tk_copy(p, pn);
        });
        float h0[4], hz[4], nb[4], o[4];
        tk_h3(h0, X[0]);
        tk_h3(hz, X[RB - 1]);
        __syncthreads();
        get(nb, bot[slot][warp]);
        tk_add(p, nb, h0);
        tk_add(o, p, x1);
        fix(std::integral_constant<int, 0>(), o, X[0]);
        tk_copy(X[0], o);
        put(top[slot ^ 1][warp], o);
        get(nb, top[slot][warp + 1]);
        tk_add(p, xz, hz);
        tk_add(o, p, nb);
        fix(std::integral_constant<int, RB - 1>(), o, X[RB - 1]);
        tk_copy(X[RB - 1], o);
        put(bot[slot ^ 1][warp + 1], o);
    };

    // One red-black half-sweep (SOR): the rows' points of one colour, in place;
    // a point reads only points of the other colour, which do not change.  PAR:
    // the parity of the band's first row; EDGE: the box may hold points that
    // keep their values.
    auto half_sweep = [&](auto par_t, auto edge_t, int slot, int yb, unsigned colin) {
        constexpr int PAR = decltype(par_t)::value;
        constexpr bool EDGE = decltype(edge_t)::value;
        constexpr bool BF = sizeof(ST) == 2;
        auto row = [&](auto i_t, const float(&n)[4], const float(&s)[4]) {
            constexpr int i = decltype(i_t)::value;
            sor_row_reg<BF, PAR ^ (i & 1), EDGE>(n, X[i], s, P.a, P.b, !EDGE || (yb + i >= 1 && yb + i <= R - 2), colin);
        };
        tk_for<1, RB - 1>([&](auto i_t) { row(i_t, X[decltype(i_t)::value - 1], X[decltype(i_t)::value + 1]); });
        __syncthreads();
        float nb[4];
        get(nb, bot[slot][warp]);
        row(std::integral_constant<int, 0>(), nb, X[1]);
        put(top[slot ^ 1][warp], X[0]);
        get(nb, top[slot][warp + 1]);
        row(std::integral_constant<int, RB - 1>(), X[RB - 2], nb);
        put(bot[slot ^ 1][warp + 1], X[RB - 1]);
    };

    LLWait wait{P.timeout_ns, P.err, false};
    for (int pass = 0; pass < P.n_pass; ++pass) {
        const bool last = pass == P.n_pass - 1;
        const int nk = last ? P.k_last : TK_HALO;
        put(top[0][warp], X[0]);
        put(bot[0][warp + 1], X[RB - 1]);
        if constexpr (SOR) {
            const TilePlace g = *where();
            const int yb = g.y0 - TK_HALO + warp * RB, gx = g.x0 - TK_HALO + lane * 4;
            const bool edge = variant || g.ty == 0 || g.ty == P.ny - 1;
            unsigned colin = 0;  // interior columns among the lane's four
#pragma unroll
            for (int e = 0; e < 4; ++e)
                if (gx + e >= 1 && gx + e <= C - 2) colin |= 1u << e;
            using Even = std::integral_constant<int, 0>;
            using Odd = std::integral_constant<int, 1>;
            using Edge = std::true_type;
            using Plain = std::false_type;
            // red (even row + column) first; x0 is even, and so is each lane's column
#pragma unroll 1
            for (int t = 0; t < nk; ++t) {
                if ((yb + t) & 1)
                    edge ? half_sweep(Odd(), Edge(), t & 1, yb, colin) : half_sweep(Odd(), Plain(), t & 1, yb, colin);
                else
                    edge ? half_sweep(Even(), Edge(), t & 1, yb, colin) : half_sweep(Even(), Plain(), t & 1, yb, colin);
            }
        } else {
            auto steps = [&](auto cf_t) {
#pragma unroll 1
                for (int t = 0; t < nk; ++t) step(cf_t, t & 1);
            };
            switch (variant) {
                case 0: steps(std::integral_constant<int, 0>()); break;
                case 1: steps(std::integral_constant<int, 1>()); break;
                case 2: steps(std::integral_constant<int, 2>()); break;
                case 3: steps(std::integral_constant<int, 3>()); break;
                case 4: steps(std::integral_constant<int, 4>()); break;
                case 5: steps(std::integral_constant<int, 5>()); break;
                default: steps(std::integral_constant<int, 6>()); break;
            }
        }
        // the box to shared memory, for Jacobi times 0.2^nk as hi + lo (the
        // product is rounded once from a ~48-bit factor)
        if constexpr (SOR) {
            tk_for<0, RB>([&](auto i_t) { put(band + decltype(i_t)::value * 32, X[decltype(i_t)::value]); });
        } else {
            const TileParams::Factor f = large ? P.factor_large[last] : P.factor[last];
            const float hi = f.hi, lo = f.lo;
            const float2 h2 = make_float2(hi, hi), l2 = make_float2(lo, lo);
            tk_for<0, RB>([&](auto i_t) {
                constexpr int i = decltype(i_t)::value;
                const float2 a = make_float2(X[i][0], X[i][1]), b = make_float2(X[i][2], X[i][3]);
                const float2 u = __ffma2_rn(a, h2, __fmul2_rn(a, l2)), v = __ffma2_rn(b, h2, __fmul2_rn(b, l2));
                band[i * 32 + lane] = make_float4(u.x, u.y, v.x, v.y);
            });
        }
        __syncthreads();
        const TilePlace g = *where();
        const int tx = g.tx, ty = g.ty;
        // the ring's exact values (SOR never changes them)
        if (!SOR && (variant || ty == 0 || ty == P.ny - 1)) {
            if (tid < BY && tx == 0) box[tid][TK_HALO] = ring_col[0][tid];
            if (tid < BY && tx == P.nx - 1) box[tid][rq] = ring_col[1][tid];
            if (tid < TK_W && ty == 0) box[TK_HALO][tid] = ring_row[0][tid];
            if (tid < TK_W && ty == P.ny - 1) box[BY - TK_HALO - 1][tid] = ring_row[1][tid];
            __syncthreads();
        }
        if (last) break;
        const uint32_t stamp = static_cast<uint32_t>(pass) + 1;
        // exchange words of this pass: rows [tile row][0 up, 1 down][8][ldx],
        // columns [tile column][0 west, 1 east][R][8]
        uint64_t *const xr = P.xrows + static_cast<size_t>(pass & 1) * P.ny * 2 * TK_HALO * P.ldx;
        uint64_t *const xc = P.xcols + static_cast<size_t>(pass & 1) * P.nx * 2 * TK_HALO * R;
        // All threads write what the neighbours need, then read the halo, in
        // one round of 16-byte accesses each: 16 rows of 64 word pairs, then 8
        // pairs for each row of the tile (4 west, 4 east).
        constexpr int NR = 2 * TK_HALO * TK_W / 2 / NT;
        constexpr int NC = (TY * TK_HALO + NT - 1) / NT;
        const int pr = tid % (TK_W / 2), hr = tid / (TK_W / 2);
        const int sd = (tid >> 2) & 1;
        const int col = g.x0 - TK_HALO + 2 * pr;
        {
            uint64_t *const rows = xr + static_cast<ptrdiff_t>(ty * 2) * TK_HALO * P.ldx + col;
            const bool own = col >= g.x0 && col < g.x1;
#pragma unroll
            for (int n = 0; n < NR; ++n) {
                const int h = n * (NT * 2 / TK_W) + hr;  // 0..7 for the tiles above, 8..15 below
                if (own && (h < TK_HALO ? ty > 0 : ty + 1 < P.ny)) {
                    const int b = (h < TK_HALO ? g.rn + h : g.rs + h - TK_HALO) - (g.y0 - TK_HALO);
                    const float2 v = *reinterpret_cast<const float2 *>(&box[b][2 * pr]);
                    ll_store(rows + static_cast<ptrdiff_t>(h) * P.ldx, v.x, v.y, stamp);
                }
            }
            const int c = sd ? g.ce : g.cw;
            uint64_t *const cols = xc + (static_cast<ptrdiff_t>(tx * 2 + sd) * R + g.y0) * TK_HALO + (tid & 3) * 2;
#pragma unroll
            for (int n = 0; n < NC; ++n) {
                const int r = n * (NT / TK_HALO) + (tid >> 3);
                if (c >= 0 && r < g.y1 - g.y0) {
                    const float2 v =
                        *reinterpret_cast<const float2 *>(&box[TK_HALO + r][TK_HALO + c - g.x0 + (tid & 3) * 2]);
                    ll_store(cols + r * TK_HALO, v.x, v.y, stamp);
                }
            }
        }
        {
            const bool col_ok = col >= 0 && col < C;
            const bool side_ok = sd ? tx + 1 < P.nx : tx > 0;
            const uint64_t *const rows = xr + static_cast<ptrdiff_t>(ty * 2 - 1) * TK_HALO * P.ldx + col;
            const uint64_t *const cols =
                xc + (static_cast<ptrdiff_t>((sd ? tx + 1 : tx - 1) * 2 + 1 - sd) * R + g.y0) * TK_HALO + (tid & 3) * 2;
            float2 v[NR + NC];
            const uint32_t expect = stamp + P.stuck;
            // (every thread loads every time, what lies off the grid from the
            // first word and unchecked: loads under conditions would wait for
            // one another)
            // (first one word pair a thread until it is there: all of them,
            // again and again, would fill L2's bandwidth before the data does)
            wait.until([&]() -> bool {
                const bool want = col_ok && ty > 0;
                const int r = tid >> 3;
                return ll_load(v[0].x, v[0].y, want ? rows + static_cast<ptrdiff_t>(hr) * P.ldx : side_ok && r < TY ? cols + r * TK_HALO : xr, expect) ||
                       !(want || (side_ok && r < TY));
            });
            wait.until([&]() -> bool {
                bool ok = true;
#pragma unroll
                for (int n = 0; n < NR; ++n) {
                    const int h = n * (NT * 2 / TK_W) + hr;  // 0..7 above, 8..15 below
                    const bool want = col_ok && (h < TK_HALO ? ty > 0 : ty + 1 < P.ny);
                    // (above: the "down" rows of tile row ty-1; below: the "up" rows of ty+1)
                    const uint64_t *const p = rows + static_cast<ptrdiff_t>(h < TK_HALO ? h : h + 2 * TK_HALO) * P.ldx;
                    ok &= ll_load(v[n].x, v[n].y, want ? p : xr, expect) || !want;
                }
#pragma unroll
                for (int n = 0; n < NC; ++n) {
                    const int r = n * (NT / TK_HALO) + (tid >> 3);
                    const bool want = side_ok && r < TY;
                    ok &= ll_load(v[NR + n].x, v[NR + n].y, want ? cols + r * TK_HALO : xr, expect) || !want;
                }
                return ok;
            });
            float m = 0.f;
#pragma unroll
            for (int n = 0; n < NR; ++n) {
                const int h = n * (NT * 2 / TK_W) + hr;
                if (h < TK_HALO ? ty > 0 : ty + 1 < P.ny) {
                    *reinterpret_cast<float2 *>(&box[h < TK_HALO ? h : h + BY - 2 * TK_HALO][2 * pr]) = v[n];
                    m = fmaxf(m, fmaxf(fabsf(v[n].x), fabsf(v[n].y)));
                }
            }
#pragma unroll
            for (int n = 0; n < NC; ++n) {
                const int r = n * (NT / TK_HALO) + (tid >> 3);
                if (side_ok && r < TY) {
                    *reinterpret_cast<float2 *>(&box[TK_HALO + r][(sd ? TK_W - TK_HALO : 0) + (tid & 3) * 2]) = v[NR + n];
                    m = fmaxf(m, fmaxf(fabsf(v[NR + n].x), fabsf(v[NR + n].y)));
                }
            }
            note_large(m);
        }
        __syncthreads();
        take_band();
    }

    const TilePlace g = *where();
    const int gx = g.x0 - TK_HALO + lane * 4;
    if (gx >= g.x0 && gx < g.x1) {  // (x0 and x1 are multiples of 4, or x1 = C)
        const bool full = gx + 4 <= C && P.vec;
        for (int r = g.y0 + warp; r < g.y1; r += NW) {
            ST *q = static_cast<ST *>(P.out) + static_cast<size_t>(r) * P.ld + gx;
            float v[4];
            get(v, reinterpret_cast<const float4 *>(box[r - g.y0 + TK_HALO]));
            if (full) {
                VecIO<ST, 4>::store(q, v);
            } else {
#pragma unroll
                for (int e = 0; e < 4; ++e)
                    if (gx + e < C) q[e] = from_ct<ST>(v[e]);
            }
        }
    }
}

template <int NW, int RB, bool SOR = false> const void *tile_fn_of(int dtype) {
    return dtype == SDFG_BF16 ? reinterpret_cast<const void *>(&tile_kernel<__nv_bfloat16, NW, RB, SOR>)
                              : reinterpret_cast<const void *>(&tile_kernel<float, NW, RB, SOR>);
}

}  // namespace sdfg
