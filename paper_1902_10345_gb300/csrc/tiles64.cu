// FP64 tiles: every step of one FP64 grid in one cooperative launch, the grid
// held in shared memory from the first step to the last (the FP64 counterpart
// of tiles.cuh).
//
// What bounds FP64 here is the FP64 pipe alone: about two lanes per SM and
// clock, so a point's five operations cost an SM 2.5 clocks and everything else
// is small beside them.  Hence the design: every SM gets an equal share of the
// grid (one tile per CTA, one CTA per SM, sizes that differ by one row or
// column at most), tiles are plain row-major arrays walked point by point so
// that no lane idles, and little is recomputed: the halo is K <= 8 cells, step
// s of a pass updates the tile and K - s cells around it, and K and the tiling
// are chosen for the grid (plan_tiles64).  Measured, against a launch per 4
// steps of the streamed kernel: 256^2 T=100 164 us (1076), 700 x 300 T=100 317
// (1079), 1000^2 T=50 573 (957), 1400^2 T=30 656 (1225): 90 of about 115
// GUpdates/s that the pipe allows at the largest, the exchange and the grid's
// small share per SM at the smallest.
//
// Every point is 0.2 * (c + ((n + s) + (w + e))), each operation rounded on its
// own: bit for bit the definition, whatever the tiling.
#include <string.h>

#include <algorithm>
#include <cmath>

#include "exchange.cuh"
#include "launchset.h"
#include "runtime.h"
#include "tiles.h"

namespace sdfg {

constexpr int T64_THREADS = 512;
constexpr int T64_MAX_K = 8;

struct Tile64Params {
    const double *in;
    double *out;
    uint64_t *words;  // exchange words [2][R][C][2], zero before the launch
    int *err;
    int R, C, ld;
    int nx, ny, K;
    int bw;           // pitch of the box
    int box;          // elements of the box
    int n_pass, k_last;
    unsigned long long timeout_ns;
    unsigned stuck;   // test hook: the halo waits are for passes that far ahead (0: none)
};

__global__ void __launch_bounds__(T64_THREADS, 1) tile64_kernel(const __grid_constant__ Tile64Params P) {
    extern __shared__ __align__(16) double smem64[];
    const int tid = threadIdx.x;
    const int tx = blockIdx.x % P.nx, ty = blockIdx.x / P.nx;
    const int R = P.R, C = P.C, K = P.K, bw = P.bw;
    const int x0 = tx * C / P.nx, x1 = (tx + 1) * C / P.nx;
    const int y0 = ty * R / P.ny, y1 = (ty + 1) * R / P.ny;
    // box element (y, x) <-> grid point (y0 - K + y, x0 - K + x)
    double *cur = smem64, *nxt = smem64 + P.box;
    auto at = [&](int r, int c) { return (r - y0 + K) * bw + (c - x0 + K); };
    // f(r, c) for the points of rows [ra, rb) x columns [ca, cb), thread by thread
    auto each = [&](int ra, int rb, int ca, int cb, auto f) {
        const unsigned w = cb - ca, n = w * (rb - ra);
        const unsigned magic = 0xffffffffu / w + 1u;  // floor(i / w) for i * w < 2^32
        for (unsigned i = tid; i < n; i += T64_THREADS) {
            const unsigned q = w == 1 ? i : __umulhi(i, magic);
            f(ra + static_cast<int>(q), ca + static_cast<int>(i - q * w));
        }
    };
    each(max(y0 - K, 0), min(y1 + K, R), max(x0 - K, 0), min(x1 + K, C), [&](int r, int c) {
        const double v = P.in[static_cast<size_t>(r) * P.ld + c];
        cur[at(r, c)] = v;
        nxt[at(r, c)] = v;  // (the boundary ring is never computed)
    });
    __syncthreads();
    LLWait wait{P.timeout_ns, P.err, false};
    for (int pass = 0; pass < P.n_pass; ++pass) {
        const bool last = pass == P.n_pass - 1;
        const int nk = last ? P.k_last : K;
        for (int s = 1; s <= nk; ++s) {
            const int h = nk - s;
            each(max(y0 - h, 1), min(y1 + h, R - 1), max(x0 - h, 1), min(x1 + h, C - 1), [&](int r, int c) {
                const int i = at(r, c);
                nxt[i] = stencil_point(cur[i], cur[i - bw], cur[i + bw], cur[i - 1], cur[i + 1]);
            });
            __syncthreads();
            double *t = cur;
            cur = nxt;
            nxt = t;
        }
        if (last) break;
        const uint32_t stamp = static_cast<uint32_t>(pass) + 1;
        uint64_t *const words = P.words + static_cast<size_t>(pass & 1) * R * C * 2;
        // what the neighbours hold as halo
        const int ra = ty > 0 ? y0 + K : y0, rb = ty + 1 < P.ny ? y1 - K : y1;
        const int ca = tx > 0 ? x0 + K : x0, cb = tx + 1 < P.nx ? x1 - K : x1;
        each(y0, y1, x0, x1, [&](int r, int c) {
            if (r < ra || r >= rb || c < ca || c >= cb)
                ll_store(words + (static_cast<size_t>(r) * C + c) * 2, cur[at(r, c)], stamp);
        });
        // the halo: the rows above and below (corners included), then the columns
        // beside the tile; four loads of a thread in flight
        const int ha = max(y0 - K, 0), hb = min(y1 + K, R), la = max(x0 - K, 0), lb = min(x1 + K, C);
        const int n_up = (y0 - ha) * (lb - la), n_dn = (hb - y1) * (lb - la);
        const int side = (x0 - la) + (lb - x1), n = n_up + n_dn + side * (y1 - y0);
        for (int i0 = 0; i0 < n; i0 += 4 * T64_THREADS) {
            double v[4];
            int to[4];
            const uint64_t *src[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                int i = i0 + q * T64_THREADS + tid, r = 0, c = 0;
                to[q] = -1;
                src[q] = words;  // past the end: any word, unchecked
                if (i < n) {
                    if (i < n_up + n_dn) {
                        r = i / (lb - la);
                        c = la + i - r * (lb - la);
                        r += r < y0 - ha ? ha : y1 - (y0 - ha);
                    } else {
                        i -= n_up + n_dn;
                        r = i / side;
                        c = i - r * side;
                        c += c < x0 - la ? la : x1 - (x0 - la);
                        r += y0;
                    }
                    to[q] = at(r, c);
                    src[q] = words + (static_cast<size_t>(r) * C + c) * 2;
                }
            }
            wait.until([&]() -> bool {
                bool ok = true;
#pragma unroll
                for (int q = 0; q < 4; ++q) ok &= ll_load(v[q], src[q], stamp + P.stuck) || to[q] < 0;
                return ok;
            });
#pragma unroll
            for (int q = 0; q < 4; ++q)
                if (to[q] >= 0) cur[to[q]] = v[q];
        }
        __syncthreads();
    }
    each(y0, y1, x0, x1, [&](int r, int c) { P.out[static_cast<size_t>(r) * P.ld + c] = cur[at(r, c)]; });
}

// ------------------------------------------------------------------ host -----
// The tiling with the least estimated time per step: the FP64 pipe's 64 clocks
// per warp and operation on the fullest scheduler, plus an exchange per K steps
// (about 1.5 us).  256^2 T=100, 8 x 19 tiles: K=1 255 us, 2 187, 3 172, 4 164,
// 6 171, 8 177; 4 x 25 to 25 x 6 tiles lie within 5% of each other.
static bool plan_tiles64(int R, int C, long long T, int sm_count, size_t smem_max, Tile64Params *best) {
    if (R < 3 || C < 3 || static_cast<long long>(R) * C > (1LL << 30)) return false;
    double best_cost = 0.0;
    for (int ny = 1; ny <= std::min(sm_count, R); ++ny) {
        const int nx = std::min(sm_count / ny, C);
        const int th = (R + ny - 1) / ny, tw = (C + nx - 1) / nx;
        if (ny > 1 && nx > 1 && (th > 8 * tw || tw > 8 * th)) continue;
        const int least = std::min(ny > 1 ? R / ny : T64_MAX_K, nx > 1 ? C / nx : T64_MAX_K);
        for (int K : {1, 2, 3, 4, 6, 8}) {
            if (K > least || (K > 1 && K > T)) break;
            const long long box = static_cast<long long>(th + 2 * K) * (tw + 2 * K);
            if (2 * box * sizeof(double) > smem_max) break;
            double warps = 0.0;  // of the fullest scheduler, over the K steps
            for (int h = 0; h < K; ++h) {
                const int w = (std::min(th + 2 * h, R) * std::min(tw + 2 * h, C) + 31) / 32;
                warps += (w + 3) / 4;
            }
            const double cost = (warps * 5 * 64 + K * 250.0 + 2800.0) / K;
            if (best_cost == 0.0 || cost < best_cost) {
                best_cost = cost;
                best->nx = nx;
                best->ny = ny;
                best->K = K;
                best->bw = tw + 2 * K;
                best->box = static_cast<int>(box);
            }
        }
    }
    return best_cost > 0.0;
}

int run_tiles64(const void *in, void *out, int R, int C, int ld, long long T, DeviceState *st, cudaStream_t s, bool *ran) {
    *ran = false;
    int smem_max = 0;
    SDFG_CUDA(cudaDeviceGetAttribute(&smem_max, cudaDevAttrMaxSharedMemoryPerBlockOptin, st->device));
    Tile64Params p;
    memset(&p, 0, sizeof(p));
    if (!plan_tiles64(R, C, T, st->sm_count, static_cast<size_t>(smem_max), &p)) return SDFG_OK;
    p.in = static_cast<const double *>(in);
    p.out = static_cast<double *>(out);
    p.err = st->d_err;
    p.R = R;
    p.C = C;
    p.ld = ld;
    p.n_pass = static_cast<int>((T + p.K - 1) / p.K);
    p.k_last = static_cast<int>(T - static_cast<long long>(p.n_pass - 1) * p.K);
    p.timeout_ns = test_hooks().timeout_ns ? test_hooks().timeout_ns : DEFAULT_TIMEOUT_NS;
    p.stuck = test_hooks().inject_stuck_wait ? LL_NEVER : 0;
    const size_t smem = 2 * sizeof(double) * static_cast<size_t>(p.box);
    const void *fn = reinterpret_cast<const void *>(&tile64_kernel);
    SDFG_CUDA(cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_max));
    // a single pass in place: a tile may not store what a neighbour still has to load
    const bool staged = in == out && p.n_pass == 1;
    const size_t words = p.n_pass > 1 ? static_cast<size_t>(4) * R * C * sizeof(uint64_t) : 0;
    const size_t bytes = staged ? static_cast<size_t>(R) * ld * sizeof(double) : words;
    void *ws = nullptr;
    int rc = scratch_alloc(&ws, bytes, s);
    if (rc == SDFG_ERR_NOMEM) return SDFG_OK;  // the caller's other path needs less
    if (rc != SDFG_OK) return rc;
    p.words = static_cast<uint64_t *>(ws);
    if (staged) p.out = static_cast<double *>(ws);
    cudaError_t e = words ? cudaMemsetAsync(ws, 0, words, s) : cudaSuccess;
    if (e == cudaSuccess) {
        void *args[] = {&p};
        TimedLaunch t = stats_begin(FAM_RESIDENT, s);
        e = cudaLaunchCooperativeKernel(fn, dim3(p.nx * p.ny), dim3(T64_THREADS), args, smem, s);
        stats_end(t, s);
    }
    if (e == cudaErrorCooperativeLaunchTooLarge) {
        cudaGetLastError();  // the tiles do not fit side by side (a partition of the device)
    } else if (e != cudaSuccess) {
        rc = cuda_error(e, "FP64 tile launch");
    } else {
        *ran = true;
        if (staged) rc = launch_copy2d(out, ld, ws, ld, R, C, SDFG_F64, s);
    }
    scratch_free(ws, s);
    return rc;
}

}  // namespace sdfg
