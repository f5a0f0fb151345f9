// K fused steps of the 3-D 7-point stencil per launch (FP32 and BF16 storage;
// StateFusion, paper App. B; see jacobi3d.cu for the method and its one-step
// kernel).
//
// A CTA of NW warps streams a column of planes: a box of NW RB rows x 128
// columns per plane, of which (NW RB - 2K) x 120 (FP32; 112 for BF16) are its
// tile and the rest the halo of K.  A lane holds 4 columns of RB rows.  Plane
// after plane arrives by TMA, NS planes ahead.  For each level l < K a lane
// keeps, for its rows, the plane of level l that came last (a) and the partial
// sum of that plane's output (p): when the next plane x comes,
//     o = p + x            (the finished plane below, level l+1)
//     p = a + (n + s) + (w + c + e)      of x
// so a plane costs one pass over the registers per level: 22 FADD and 2 SHFL
// for 4 points.  All levels' o come first: they need no neighbour, each one
// add after the level below.  Only then the p: level 0 reads the rows above and
// below from the TMA box, for the others a warp passes its first and last row
// to its neighbours through shared memory, all levels at once, with one barrier
// per plane.
//
// Arithmetic as in the 2-D units (level_p in temporal_unit.cuh): sums carried
// unscaled, 7^-K applied once as hi + lo.  So that nothing overflows that does not
// in the plain order, level 0 makes its sums 8^-(K-1) of what they are (a power of
// two, inside multiply-adds: 2 products more per 4 points): level l > 0 holds 7^l
// 8^(1-K) times the state, at most 7 times at the end, and loses no bit of values
// above 2^-117.  hi is rounded down, which makes lo positive: an infinity times
// either keeps its sign.  The fixed shell is held scaled like every other value
// (times 7 at each level) and never stored: j3_shell_copy puts it into both
// ping-pong boxes.
//
// What bounds it: one step per launch is bound by HBM (8 bytes per FP32 update:
// 512^3 at 172 us per step, 0.9 of the measured bandwidth).  Here it is issue:
// about 40 instructions per 4 points and level, of which 24 are the arithmetic,
// at 59% of the issue slots, on 1.75 times the points (in the plane 1.59: 5 tile
// columns of 128 lanes and 18 tile rows of 36 for 510 x 510; along z 1.10: 2K planes
// of every run and the last wave); DRAM is at 30%.
// Measured on 512^3, us per step, warps x rows: K=2 16x3 107, 12x5 106; K=3
// 12x3 100, 8x5 117, 16x2 125, 12x4 and 8x6 spill (115, 122); K=4 8x4 113.
#include <math.h>
#include <string.h>

#include <algorithm>
#include <type_traits>

#include "device_common.cuh"
#include "jacobi3d.h"
#include "runtime.h"

namespace sdfg {

constexpr int JF_NS = 4;  // ring stages (planes)

template <int I, int N, class F> __device__ __forceinline__ void jf_for(F &&f) {
    if constexpr (I < N) {
        f(std::integral_constant<int, I>());
        jf_for<I + 1, N>(f);
    }
}

// (Scalar adds: packed FP32x2 ones issue half as often but need their operands
// in register pairs; 109 against 100 us per step on 512^3.)
__device__ __forceinline__ void jf_add(float (&o)[4], const float (&a)[4], const float (&b)[4]) {
#pragma unroll
    for (int e = 0; e < 4; ++e) o[e] = __fadd_rn(a[e], b[e]);
}

template <class ST, int K, int NW, int RB>
__global__ void __launch_bounds__(32 * NW, 1) jacobi3d_fused_kernel(const __grid_constant__ CUtensorMap tm, ST *dst,
                                                                    const J3FGeo g, float hi, float lo, int *err,
                                                                    unsigned long long timeout_ns) {
    constexpr int W = 128;
    constexpr int BY = NW * RB;
    constexpr int TY = BY - 2 * K;
    constexpr int XH = 16 / sizeof(ST);  // column halo: 16 bytes, so the box start stays TMA-aligned
    constexpr int TX = W - 2 * XH;
    static_assert(XH >= K && TY > 0 && BY <= 256, "halo");
    static_assert(RB <= 3, "(RB - 1) ld fits 32 unsigned bits");
    constexpr float DOWN = 1.0f / (1 << 3 * (K - 1));  // of level 0's sums
    constexpr uint32_t PLANE_BYTES = BY * W * sizeof(ST);
    extern __shared__ __align__(128) unsigned char smem_raw[];
    __shared__ __align__(8) uint64_t bars[JF_NS];
    // first and last rows of the bands, per level (from 1) and plane parity; the rows
    // beyond the box (top[..][NW], bot[..][0]) may hold anything finite
    __shared__ __align__(16) float4 top[2][K - 1][NW + 1][32];
    __shared__ __align__(16) float4 bot[2][K - 1][NW + 1][32];
    ST *ring = reinterpret_cast<ST *>(smem_raw);

    const int tid = threadIdx.x;
    const int lane = tid & 31;
    const int warp = tid >> 5;
    int b = blockIdx.x;
    const int tx = b % g.tiles_x;
    b /= g.tiles_x;
    const int ty = b % g.tiles_y;
    const int zs = b / g.tiles_y;
    const int x0 = tx * TX, y0 = ty * TY;
    const int z0 = zs * g.zseg, z1 = min(z0 + g.zseg, g.D);
    const int n_planes = z1 - z0 + 2 * K;  // input planes z0-K .. z1+K-1

    if (tid == 0) {
        for (int s = 0; s < JF_NS; ++s) mbar_init(&bars[s], 1);
        mbar_init_fence();
        tmap_prefetch(&tm);
    }
    if (warp == 0) {
        const float4 z = make_float4(0.f, 0.f, 0.f, 0.f);
        for (int q = 0; q < 2; ++q)
            for (int l = 0; l < K - 1; ++l) bot[q][l][0][lane] = top[q][l][NW][lane] = z;
    }
    __syncthreads();
    auto issue = [&](int m) {
        const int st = m % JF_NS;
        mbar_arrive_expect_tx(&bars[st], PLANE_BYTES);
        tma_load_3d(ring + st * (BY * W), &tm, x0 - XH, y0 - K, z0 - K + m, &bars[st]);
    };
    if (tid == 0)
        for (int m = 0; m < min(JF_NS, n_planes); ++m) issue(m);

    const int gx = x0 - XH + lane * 4;          // grid column of element 0
    const int yb = y0 - K + warp * RB;          // grid row of the band's first row
    unsigned colmask = 0;                       // shell columns (and columns off the grid) among the four
#pragma unroll
    for (int e = 0; e < 4; ++e)
        if (gx + e <= 0 || gx + e >= g.C - 1) colmask |= 1u << e;
    const bool own_cols = lane * 4 >= XH && lane * 4 < XH + TX && gx < g.C - 1;
    // Which shell points this warp's band holds, beside those of shell planes:
    // 0 none, 1 column 0 (element 0 of one lane), 2 both columns, 3 also rows,
    // 4 + e column C-1 (element e of one lane).
    // Points off the grid may take any value: they reach the interior only
    // through the shell.
    const bool row_shell = (yb <= 0 && yb + RB > 0) || (yb <= g.R - 1 && yb + RB > g.R - 1);
    const int rq = g.C - 1 - (x0 - XH);  // box column of column C-1
    const int var = row_shell ? 3 : rq >= W ? (x0 == 0 ? 1 : 0) : x0 == 0 ? 2 : 4 + (rq & 3);
    const bool lane_l = lane == XH / 4, lane_r = lane == (rq >> 2);
    unsigned store_rows = 0;  // the band's rows that are stored
#pragma unroll
    for (int i = 0; i < RB; ++i) {
        const int br = warp * RB + i;
        if (br >= K && br < BY - K && yb + i >= 1 && yb + i <= g.R - 2) store_rows |= 1u << i;
    }

    float A[2][K][RB][4];  // by plane parity: the plane of level l that came last, and the one before
    float P[K][RB][4];
    jf_for<0, K>([&](auto l_t) {
        constexpr int l = decltype(l_t)::value;
        jf_for<0, RB>([&](auto i_t) {
            constexpr int i = decltype(i_t)::value;
#pragma unroll
            for (int e = 0; e < 4; ++e) A[0][l][i][e] = A[1][l][i][e] = P[l][i][e] = 0.f;
        });
    });
    bool dead = false;  // a wait ran out
    ST *out = dst + static_cast<long long>(z0 - 2 * K) * g.plane + static_cast<long long>(yb) * g.ld + gx;

    // One input plane m of parity Q.  (The warps of a CTA run different
    // variants of it: the barrier is the same.)
    auto plane = [&](auto q_t, auto var_t, int m) {
        constexpr int Q = decltype(q_t)::value;
        constexpr int VAR = decltype(var_t)::value;
        const int zi = z0 - K + m;  // its global index; level l receives plane zi - l
        const ST *box = ring + (m % JF_NS) * (BY * W) + lane * 4;
        jf_for<0, RB>([&](auto i_t) {
            constexpr int i = decltype(i_t)::value;
            VecIO<ST, 4>::load(A[Q][0][i], box + (warp * RB + i) * W);
        });
        float north[4], south[4];
        VecIO<ST, 4>::load(north, box + max(warp * RB - 1, 0) * W);
        VecIO<ST, 4>::load(south, box + min(warp * RB + RB, BY - 1) * W);
        // rows of the plane that the last level finishes
        const unsigned rows = m >= 2 * K && zi - K >= 1 && zi - K <= g.D - 2 && own_cols ? store_rows : 0u;
        // all levels' finished planes: one add each, no neighbour
        jf_for<0, K>([&](auto l_t) {
            constexpr int l = decltype(l_t)::value;
            jf_for<0, RB>([&](auto i_t) {
                constexpr int i = decltype(i_t)::value;
                const float(&a)[4] = A[Q ^ 1][l][i];
                constexpr float SEVEN = l == 0 ? 7.0f * DOWN : 7.0f;
                float o[4];
                if constexpr (l == 0) {
#pragma unroll
                    for (int e = 0; e < 4; ++e) o[e] = __fmaf_rn(A[Q][l][i][e], DOWN, P[l][i][e]);
                } else {
                    jf_add(o, P[l][i], A[Q][l][i]);
                }
                if constexpr (VAR == 1) {
                    if (lane_l) o[0] = __fmul_rn(SEVEN, a[0]);
                }
                if constexpr (VAR >= 4) {
                    if (lane_r) o[VAR - 4] = __fmul_rn(SEVEN, a[VAR - 4]);
                }
                if constexpr (VAR == 2 || VAR == 3) {
                    const int zc = zi - l - 1, r = yb + i;  // the plane this level finishes
                    const unsigned m4 = VAR == 3 && (zc <= 0 || zc >= g.D - 1 || r <= 0 || r >= g.R - 1) ? 15u : colmask;
#pragma unroll
                    for (int e = 0; e < 4; ++e)
                        if ((m4 >> e) & 1u) o[e] = __fmul_rn(SEVEN, a[e]);
                }
                if constexpr (l + 1 < K) {
#pragma unroll
                    for (int e = 0; e < 4; ++e) A[Q][l + 1][i][e] = o[e];
                } else {
                    const float2 u = make_float2(o[0], o[1]), v = make_float2(o[2], o[3]);
                    const float2 f = __ffma2_rn(u, make_float2(hi, hi), __fmul2_rn(u, make_float2(lo, lo)));
                    const float2 h2 = __ffma2_rn(v, make_float2(hi, hi), __fmul2_rn(v, make_float2(lo, lo)));
                    const float w[4] = {f.x, f.y, h2.x, h2.y};
                    // (a row of the band is at most two pitches off: 32 unsigned bits hold that)
                    ST *p = out + static_cast<unsigned>(i) * static_cast<unsigned>(g.ld);
                    const int pred = rows & (1u << i);
                    if constexpr (VAR == 0) {
                        store_pred(p, w, pred);
                    } else {
                        store_pred(p, w, colmask == 0 ? pred : 0);
                        if (pred && colmask != 0) {
#pragma unroll
                            for (int e = 0; e < 4; ++e)
                                if (!((colmask >> e) & 1u)) p[e] = from_ct<ST>(w[e]);
                        }
                    }
                }
            });
            if constexpr (l > 0) {
                top[Q][l - 1][warp][lane] = make_float4(A[Q][l][0][0], A[Q][l][0][1], A[Q][l][0][2], A[Q][l][0][3]);
                bot[Q][l - 1][warp + 1][lane] =
                    make_float4(A[Q][l][RB - 1][0], A[Q][l][RB - 1][1], A[Q][l][RB - 1][2], A[Q][l][RB - 1][3]);
            }
        });
        // the partial sums for the next plane
        jf_for<0, K>([&](auto l_t) {
            constexpr int l = decltype(l_t)::value;
            const float(&x)[RB][4] = A[Q][l];
            if constexpr (l == 1) {
                asm volatile("bar.sync 0;" ::: "memory");
                // (every warp has read plane m's stage: refill it)
                if (tid == 0 && m + JF_NS < n_planes) issue(m + JF_NS);
            }
            if constexpr (l > 0) {
                const float4 n4 = bot[Q][l - 1][warp][lane], s4 = top[Q][l - 1][warp + 1][lane];
                north[0] = n4.x, north[1] = n4.y, north[2] = n4.z, north[3] = n4.w;
                south[0] = s4.x, south[1] = s4.y, south[2] = s4.z, south[3] = s4.w;
            }
            jf_for<0, RB>([&](auto i_t) {
                constexpr int i = decltype(i_t)::value;
                const float left = __shfl_up_sync(FULL_MASK, x[i][3], 1);
                const float right = __shfl_down_sync(FULL_MASK, x[i][0], 1);
                // (x + y, level 0: x DOWN + y, with y scaled already)
                auto plus = [](float u, float v) { return l == 0 ? __fmaf_rn(u, DOWN, v) : __fadd_rn(u, v); };
                float q0 = __fadd_rn(x[i][0], x[i][1]), q1 = __fadd_rn(x[i][2], x[i][3]);
                if constexpr (l == 0) q0 = __fmul_rn(q0, DOWN), q1 = __fmul_rn(q1, DOWN);
                const float h[4] = {plus(left, q0), plus(x[i][2], q0), plus(x[i][1], q1), plus(right, q1)};
                float t[4];
                float n[4], s[4];
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    n[e] = i == 0 ? north[e] : x[i == 0 ? 0 : i - 1][e];
                    s[e] = i == RB - 1 ? south[e] : x[i == RB - 1 ? 0 : i + 1][e];
                }
                jf_add(t, n, s);
                jf_add(t, t, A[Q ^ 1][l][i]);
#pragma unroll
                for (int e = 0; e < 4; ++e) P[l][i][e] = plus(t[e], h[e]);
            });
        });
        out += g.plane;
    };
    // planes [from, to), an even number of them but at the end
    auto stream = [&](auto var_t, int from, int to) {
        auto advance = [&](auto q_t, int m) {
            if (!dead && !mbar_wait_bounded(&bars[m % JF_NS], (m / JF_NS) & 1u, timeout_ns)) {
                dead = true;
                set_device_error(err, DEV_ERR_TIMEOUT_TMA);
            }
            __syncwarp();
            plane(q_t, var_t, m);
        };
#pragma unroll 1
        for (int m = from; m < to; m += 2) {
            advance(std::integral_constant<int, 0>(), m);
            if (m + 1 < to) advance(std::integral_constant<int, 1>(), m + 1);
        }
    };
    // The planes for which some level finishes a shell plane (or one off the
    // box) run the variant that tests for it, at the ends of the box only.
    int ma = min(n_planes, max(0, (2 * K + 2 - z0) & ~1));
    int mb = max(ma, min(n_planes, (g.D - z0 + K) & ~1));
    if (n_planes - mb < 2 && g.D - z0 + K >= n_planes) mb = n_planes;
    if (var == 3) ma = mb = 0;
    using V0 = std::integral_constant<int, 0>;
    using V1 = std::integral_constant<int, 1>;
    using V2 = std::integral_constant<int, 2>;
    using V3 = std::integral_constant<int, 3>;
    if (ma > 0) stream(V3(), 0, ma);
    switch (var) {
        case 0: stream(V0(), ma, mb); break;
        case 1: stream(V1(), ma, mb); break;
        case 2: stream(V2(), ma, mb); break;
        case 4: stream(std::integral_constant<int, 4>(), ma, mb); break;
        case 5: stream(std::integral_constant<int, 5>(), ma, mb); break;
        case 6: stream(std::integral_constant<int, 6>(), ma, mb); break;
        case 7: stream(std::integral_constant<int, 7>(), ma, mb); break;
        default: break;
    }
    if (mb < n_planes) stream(V3(), mb, n_planes);
    // no copy may land after the CTA has left
    if (__syncthreads_or(dead) && tid == 0)
        for (int m = max(0, n_planes - JF_NS); m < n_planes; ++m)
            mbar_wait_bounded(&bars[m % JF_NS], (m / JF_NS) & 1u, 1000000ull);
}

// The shell of a box into one or two others of the same layout.
// A warp per item: a row of the end planes, a first or last row of a plane between,
// or 256 rows of such a plane's first and last columns.  (The end planes are as large as
// the box is shallow: by 4 blocks each they took 40 us of 61 for 2 steps of 24 x 400 x 400.)
constexpr int J3_SHELL_ROWS = 256;
template <class ST>
__global__ void __launch_bounds__(256) j3_shell_kernel(const ST *__restrict__ src, ST *__restrict__ d0, ST *__restrict__ d1, int D,
                                                       int R, int C, int ld) {
    const int lane = threadIdx.x & 31;
    auto copy = [&](long long at) {
        const ST v = src[at];
        d0[at] = v;
        if (d1) d1[at] = v;
    };
    const int parts = (R - 2 + J3_SHELL_ROWS - 1) / J3_SHELL_ROWS;
    const long long n_rows = 2LL * R + 2LL * (D - 2), n = n_rows + static_cast<long long>(D - 2) * parts;
    const long long plane = static_cast<long long>(R) * ld;
    for (long long i = blockIdx.x * 8LL + (threadIdx.x >> 5); i < n; i += gridDim.x * 8LL) {
        if (i < n_rows) {
            const long long j = i - 2LL * R;  // (row within the end planes if negative)
            const long long z = j < 0 ? (i < R ? 0 : D - 1) : 1 + j / 2;
            const long long r = j < 0 ? (i < R ? i : i - R) : j % 2 ? R - 1 : 0;
            const long long at = z * plane + r * ld;
#pragma unroll 4
            for (int c = lane; c < C; c += 32) copy(at + c);
        } else {
            const long long j = i - n_rows;
            const int r0 = 1 + static_cast<int>(j % parts) * J3_SHELL_ROWS, r1 = min(r0 + J3_SHELL_ROWS, R - 1);
            const long long at = (1 + j / parts) * plane;
#pragma unroll 4
            for (int r = r0 + lane; r < r1; r += 32) {
                copy(at + static_cast<long long>(r) * ld);
                copy(at + static_cast<long long>(r) * ld + C - 1);
            }
        }
    }
}

int j3_shell_copy(const void *src, void *d0, void *d1, int D, int R, int C, int ld, int dtype, cudaStream_t s) {
    const long long items = 2LL * R + 2LL * D + static_cast<long long>(D) * ((R + J3_SHELL_ROWS - 1) / J3_SHELL_ROWS);
    const unsigned blocks = static_cast<unsigned>(std::min<long long>((items + 7) / 8, 1 << 14));
    if (dtype == SDFG_F32)
        j3_shell_kernel<float><<<blocks, 256, 0, s>>>(static_cast<const float *>(src), static_cast<float *>(d0),
                                                      static_cast<float *>(d1), D, R, C, ld);
    else
        j3_shell_kernel<__nv_bfloat16><<<blocks, 256, 0, s>>>(static_cast<const __nv_bfloat16 *>(src),
                                                              static_cast<__nv_bfloat16 *>(d0),
                                                              static_cast<__nv_bfloat16 *>(d1), D, R, C, ld);
    const cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? SDFG_OK : cuda_error(e, "jacobi3d shell copy");
}

// ------------------------------------------------------------------ host -----
namespace {
struct Shape {
    int K, NW, RB;
};
template <int K, int NW, int RB> const void *fn_of(int dtype) {
    return dtype == SDFG_F32 ? reinterpret_cast<const void *>(&jacobi3d_fused_kernel<float, K, NW, RB>)
                             : reinterpret_cast<const void *>(&jacobi3d_fused_kernel<__nv_bfloat16, K, NW, RB>);
}
Shape shape_of(int K) { return K == 3 ? Shape{3, 12, 3} : Shape{2, 16, 3}; }
const void *fused_fn(int K, int dtype) { return K == 3 ? fn_of<3, 12, 3>(dtype) : fn_of<2, 16, 3>(dtype); }
}  // namespace

int j3_fused_rows(int K) { return shape_of(K).NW * shape_of(K).RB; }
int j3_fused_cols() { return 128; }

// Planes per CTA: the number of runs along z for which the waves of one CTA
// per SM, each run with 2K planes of its own on top, take the fewest planes.
J3FGeo j3_fused_plan(int K, int D, int R, int C, int ld, int dtype, int sm_count) {
    J3FGeo g;
    g.D = D;
    g.R = R;
    g.C = C;
    g.ld = ld;
    g.plane = static_cast<long long>(R) * ld;
    const int TX = 128 - 2 * (16 / dtype_bytes(dtype)), TY = j3_fused_rows(K) - 2 * K;
    g.tiles_x = (C + TX - 1) / TX;
    g.tiles_y = (R + TY - 1) / TY;
    const long long tiles = static_cast<long long>(g.tiles_x) * g.tiles_y;
    long long best = 0;
    g.n_zseg = 1;
    for (int n = 1; n <= std::min(D, 512); ++n) {
        const long long waves = (tiles * n + sm_count - 1) / sm_count;
        const long long cost = waves * ((D + n - 1) / n + 2 * K + 2);
        if (n == 1 || cost < best) {
            best = cost;
            g.n_zseg = n;
        }
    }
    g.zseg = (D + g.n_zseg - 1) / g.n_zseg;
    g.n_zseg = (D + g.zseg - 1) / g.zseg;
    return g;
}

int launch_j3_fused(const CUtensorMap &tm, void *dst, const J3FGeo &g, int K, int dtype, int *err, cudaStream_t s) {
    const void *fn = fused_fn(K, dtype);
    const size_t smem = static_cast<size_t>(JF_NS) * j3_fused_rows(K) * 128 * dtype_bytes(dtype);
    int rc = raise_smem_limit(fn, smem);
    if (rc != SDFG_OK) return rc;
    double f = ldexp(1.0, 3 * (K - 1));
    for (int i = 0; i < K; ++i) f /= 7.0;
    float hi = static_cast<float>(f);
    if (hi > f) hi = nextafterf(hi, 0.0f);
    float lo = static_cast<float>(f - static_cast<double>(hi));
    CUtensorMap t = tm;
    J3FGeo gg = g;
    void *dp = dst;
    unsigned long long to = DEFAULT_TIMEOUT_NS;
    void *args[] = {&t, &dp, &gg, &hi, &lo, &err, &to};
    const unsigned blocks = static_cast<unsigned>(static_cast<long long>(g.tiles_x) * g.tiles_y * g.n_zseg);
    TimedLaunch tl = stats_begin(FAM_STENCIL3D, s);
    const cudaError_t e = cudaLaunchKernel(fn, dim3(blocks), dim3(32 * shape_of(K).NW), args, smem, s);
    stats_end(tl, s);
    return e == cudaSuccess ? SDFG_OK : cuda_error(e, "jacobi3d fused launch");
}

}  // namespace sdfg
