// Single-grid entry points: sdfg_jacobi2d, _ex, _cfg, _host.
//
// The timestep loop is a sequence of passes (paper Fig. 1: a state loop whose
// body is a map; App. B StateFusion fuses k states into one pass).  Pass p
// reads buffer src_p and writes dst_p; the buffers alternate between the
// caller's `out` and one scratch grid, arranged so that the last pass writes
// `out` whenever `in` and `out` differ.
#include <string.h>

#include <algorithm>
#include <mutex>

#include "autotune.h"
#include "launchset.h"
#include "runtime.h"
#include "tiles.h"

namespace sdfg {

int validate_grid(const void *in, const void *out, int R, int C, int ld, long long T, int dtype, const char *who) {
    if (!dtype_valid(dtype)) return set_error(SDFG_ERR_INVAL, "%s: unknown dtype %d", who, dtype);
    if (R < 0 || C < 0) return set_error(SDFG_ERR_INVAL, "%s: rows=%d cols=%d must be >= 0", who, R, C);
    if (T < 0) return set_error(SDFG_ERR_INVAL, "%s: T=%lld must be >= 0", who, T);
    if (R > 0 && C > 0) {
        if (ld < C) return set_error(SDFG_ERR_INVAL, "%s: ld=%d < cols=%d", who, ld, C);
        if (!in || !out) return set_error(SDFG_ERR_INVAL, "%s: null grid pointer", who);
        const size_t S = dtype_bytes(dtype);
        const char *a = static_cast<const char *>(in);
        const char *b = static_cast<const char *>(out);
        const size_t span = (static_cast<size_t>(R - 1) * ld + C) * S;
        if (a != b && a < b + span && b < a + span)
            return set_error(SDFG_ERR_INVAL, "%s: in and out overlap without being the same grid", who);
        if (reinterpret_cast<uintptr_t>(in) % S || reinterpret_cast<uintptr_t>(out) % S)
            return set_error(SDFG_ERR_INVAL, "%s: grid pointers must be aligned to the element size", who);
    }
    return SDFG_OK;
}

// use_tuned: what the autotuner chose for the shape's class counts (not for its own trials).
int resolve_config(const sdfg_config *cfg, int R, int C, int dtype, bool use_tuned, sdfg_config *out) {
    sdfg_config c = {SDFG_KERNEL_AUTO, 0, 0, 0};
    if (cfg) c = *cfg;
    if (c.kernel < SDFG_KERNEL_AUTO || c.kernel > SDFG_KERNEL_SKEWED)
        return set_error(SDFG_ERR_INVAL, "unknown kernel family %d", c.kernel);
    if (c.k != 0 && !depth_supported(c.k)) return set_error(SDFG_ERR_INVAL, "k=%d not supported (1, 2, 4, 8)", c.k);
    if (c.seg_rows < 0 || c.warps < 0 || c.warps > MAX_WARPS)
        return set_error(SDFG_ERR_INVAL, "bad seg_rows/warps (%d/%d)", c.seg_rows, c.warps);
    sdfg_config tuned;
    const bool have = use_tuned && autotune_lookup(R, C, dtype, &tuned) && tuned.kernel != SDFG_KERNEL_AUTO;
    // large grids: one launch for all passes (no per-pass tail) -- the chain
    // kernel -- for FP32/BF16 storage; one step per launch for FP64, which the
    // FP64 pipe bounds, so that fused steps only recompute halos (2048^2 T=20
    // 867 us against 2573 for the persistent kernel, 1369 for a launch per 4
    // steps; 4096 x 4000 T=10 1622 against 2170, 2025); small grids: one
    // launch per pass
    if (c.kernel == SDFG_KERNEL_AUTO) {
        const bool large = static_cast<long long>(R) * C >= (1LL << 20);
        c.kernel = have    ? tuned.kernel
                   : large ? (dtype == SDFG_F64 ? SDFG_KERNEL_NAIVE : SDFG_KERNEL_SKEWED)
                           : SDFG_KERNEL_TEMPORAL;
    }
    if (c.k == 0) c.k = have && tuned.k ? tuned.k : default_depth(dtype);
    if (c.warps == 0) c.warps = have && tuned.warps ? tuned.warps : 4;
    if (c.seg_rows == 0 && have) c.seg_rows = tuned.seg_rows;
    *out = c;
    return SDFG_OK;
}

// Run the passes `ks` on (src0 -> ... ) alternating between buffers `first`
// and `second`; returns the buffer holding the result in *final.
static int run_pass_sequence(const void *src0, void *first, void *second, const std::vector<int> &ks, int R, int C,
                             int ld, int dtype, const sdfg_config &c, DeviceState *st, cudaStream_t s,
                             void **final) {
    *final = const_cast<void *>(src0);
    if (ks.empty()) return SDFG_OK;
    if (c.kernel == SDFG_KERNEL_RESIDENT) return run_resident_passes(src0, first, second, ks, R, C, ld, dtype, st, s, final);
    if (c.kernel == SDFG_KERNEL_NAIVE) {
        const void *src = src0;
        void *dst = first;
        for (size_t p = 0; p < ks.size(); ++p) {
            for (int t = 0; t < ks[p]; ++t) {
                int rc = launch_naive_step(src, dst, R, C, ld, dtype, s);
                if (rc != SDFG_OK) return rc;
                src = dst;
                dst = (dst == first) ? second : first;
            }
        }
        *final = const_cast<void *>(src);
        return SDFG_OK;
    }
    const int S = dtype_bytes(dtype);
    const int W = 32 * lane_cols(S);
    const int bps = std::max(1, temporal_blocks_per_sm(dtype, c.k, c.warps));
    const GridGeo g = plan_geometry(R, C, ld, dtype, c.k, c.seg_rows, static_cast<long long>(st->sm_count) * bps * c.warps);
    alignas(64) CUtensorMap tm_src0, tm_first, tm_second;
    int rc = encode_tmap(&tm_src0, src0, dtype, R, C, ld, W);
    if (rc == SDFG_OK) rc = encode_tmap(&tm_first, first, dtype, R, C, ld, W);
    if (rc == SDFG_OK) rc = encode_tmap(&tm_second, second, dtype, R, C, ld, W);
    if (rc != SDFG_OK) return rc;
    const CUtensorMap *tm_src = &tm_src0;
    void *dst = first;
    for (size_t p = 0; p < ks.size(); ++p) {
        rc = launch_temporal_pass(tm_src, dst, g, dtype, ks[p], c.warps, 0, nullptr, st->d_err, DEFAULT_TIMEOUT_NS, s);
        if (rc != SDFG_OK) return rc;
        *final = dst;
        tm_src = (dst == first) ? &tm_first : &tm_second;
        dst = (dst == first) ? second : first;
    }
    return SDFG_OK;
}

int enqueue_persistent(LaunchSet &ls, DeviceState *st, cudaStream_t s);

// ---- single grid through the persistent kernel ------------------------------
// Uploaded launch plans are kept for repeated calls with the same arguments
// (pointers, shape, T, configuration): a repeat only resets the plan's
// counters and launches.  At most kSingleCacheSize plans (and their scratch
// grids) are kept per process.
namespace {
struct SingleKey {
    const void *in;
    void *out;
    int R, C, ld, dtype, k, warps, seg_rows, device;
    long long T;
    bool operator==(const SingleKey &o) const {
        return in == o.in && out == o.out && R == o.R && C == o.C && ld == o.ld && dtype == o.dtype && k == o.k &&
               warps == o.warps && seg_rows == o.seg_rows && device == o.device && T == o.T;
    }
};
struct SingleEntry {
    SingleKey key;
    LaunchSet ls;
    void *scratch = nullptr;
    int last = 0;  // buffer holding the result
    unsigned long long stamp = 0;
};
constexpr size_t kSingleCacheSize = 8;
std::mutex g_single_mu;
std::vector<SingleEntry *> g_single;
unsigned long long g_single_clock = 0;
}  // namespace

static int run_single_persistent(const void *in, void *out, int R, int C, int ld, long long T, int dtype,
                                 const sdfg_config &c, DeviceState *st, cudaStream_t s) {
    std::lock_guard<std::mutex> lk(g_single_mu);
    const SingleKey key{in, out, R, C, ld, dtype, c.k, c.warps, c.seg_rows, st->device, T};
    SingleEntry *e = nullptr;
    for (SingleEntry *x : g_single)
        if (x->key == key) e = x;
    if (!e) {
        if (g_single.size() >= kSingleCacheSize) {
            // the evicted plan's last launch may run on another stream
            cudaDeviceSynchronize();
            auto it = std::min_element(g_single.begin(), g_single.end(),
                                       [](SingleEntry *a, SingleEntry *b) { return a->stamp < b->stamp; });
            (*it)->ls.release(s);
            scratch_free((*it)->scratch, s);
            delete *it;
            g_single.erase(it);
        }
        e = new SingleEntry();
        e->key = key;
        int rc = scratch_alloc(&e->scratch, static_cast<size_t>(R) * ld * dtype_bytes(dtype), s);
        GridRun r;
        r.buf[0] = out;
        r.buf[1] = e->scratch;
        r.buf[2] = in == out ? nullptr : const_cast<void *>(in);
        r.cur = in == out ? 0 : 2;
        r.ld = ld;
        r.R = R;
        r.C = C;
        r.steps = static_cast<int>(T);
        r.T_cap = static_cast<int>(T);
        r.seg_rows = c.seg_rows;
        e->ls.dtype = dtype;
        e->ls.k = c.k;
        e->ls.warps = c.warps;
        if (rc == SDFG_OK) rc = e->ls.build(std::vector<GridRun>(1, r));
        if (rc == SDFG_OK) rc = e->ls.upload(s);
        if (rc != SDFG_OK) {
            e->ls.release(s);
            scratch_free(e->scratch, s);
            delete e;
            return rc;
        }
        e->last = e->ls.last_dst[0];
        g_single.push_back(e);
    }
    e->stamp = ++g_single_clock;
    int rc = enqueue_persistent(e->ls, st, s);
    if (rc == SDFG_OK && e->last != 0) rc = launch_copy2d(out, ld, e->scratch, ld, R, C, dtype, s);
    return rc;
}

// Core single-grid run.  in_disposable: `in` may be overwritten (it then
// serves as the scratch grid).  use_tuned: see resolve_config.
int run_single(const void *in, void *out, int R, int C, int ld, long long T, int dtype, const sdfg_config *cfg,
               bool in_disposable, cudaStream_t s, bool use_tuned = true) {
    if (R == 0 || C == 0) return SDFG_OK;
    DeviceState *st = nullptr;
    int rc = current_device(&st);
    if (rc != SDFG_OK) return rc;
    if (T == 0 || R < 3 || C < 3) return launch_copy2d(out, ld, in, ld, R, C, dtype, s);
    sdfg_config c;
    rc = resolve_config(cfg, R, C, dtype, use_tuned, &c);
    if (rc != SDFG_OK) return rc;
    // nothing asked for, and nothing else tuned: a grid that the chip's
    // registers hold runs there from the first step to the last.  Measured
    // against the launches below (their defaults): 256^2 T=100 50 us (233, a
    // launch per pass), 1301 x 1777 on an odd pitch T=150 148 us (478),
    // 2048^2 T=1024 1345 us (6676, chains; 1610 with register-resident passes)
    sdfg_config tuned;
    if ((!cfg || (cfg->kernel == SDFG_KERNEL_AUTO && cfg->k == 0 && cfg->seg_rows == 0 && cfg->warps == 0)) &&
        (!use_tuned || !autotune_lookup(R, C, dtype, &tuned) || tuned.kernel == SDFG_KERNEL_AUTO)) {
        if (dtype == SDFG_F64) {
            bool ran = false;
            rc = run_tiles64(in, out, R, C, ld, T, st, s, &ran);
            if (rc != SDFG_OK || ran) return rc;
        }
        TilePlan plan;
        if (plan_tiles(R, C, dtype, st, &plan)) {
            rc = run_tiles(in, out, R, C, ld, T, dtype, plan, st, s);
            if (rc != SDFG_ERR_NOMEM) return rc;
        }
    }
    if (c.kernel == SDFG_KERNEL_RESIDENT && !resident_supported(dtype)) c.kernel = SDFG_KERNEL_TEMPORAL;
    const std::vector<int> ks = c.kernel == SDFG_KERNEL_NAIVE      ? std::vector<int>(1, static_cast<int>(T))
                                : c.kernel == SDFG_KERNEL_RESIDENT ? plan_resident_passes(T, c.k)
                                                                   : plan_passes(T, c.k);
    const long long n_steps_total = c.kernel == SDFG_KERNEL_NAIVE ? T : static_cast<long long>(ks.size());
    const int S = dtype_bytes(dtype);
    const bool tma_ok = tma_compatible(in, ld, dtype) && tma_compatible(out, ld, dtype);
    if (c.kernel == SDFG_KERNEL_PERSISTENT && tma_ok) {
        sdfg_config pc = c;
        if (pc.seg_rows == 0) pc.seg_rows = 128;
        if (pc.warps > 4) pc.warps = 4;
        return run_single_persistent(in, out, R, C, ld, T, dtype, pc, st, s);
    }
    if (c.kernel == SDFG_KERNEL_SKEWED && tma_ok)
        return run_single_chain(in, out, R, C, ld, T, dtype, c.k, c.seg_rows, 0, st, s);
    if (c.kernel == SDFG_KERNEL_PERSISTENT || c.kernel == SDFG_KERNEL_SKEWED) c.kernel = SDFG_KERNEL_TEMPORAL;

    if (c.kernel != SDFG_KERNEL_NAIVE && !tma_ok) {
        // stage through two aligned pitched grids
        const int ldp = (C + 31) / 32 * 32;
        void *a = nullptr, *b = nullptr;
        const size_t bytes = static_cast<size_t>(R) * ldp * S;
        rc = scratch_alloc(&a, bytes, s);
        if (rc == SDFG_OK) rc = scratch_alloc(&b, bytes, s);
        void *fin = nullptr;
        if (rc == SDFG_OK) rc = launch_copy2d(a, ldp, in, ld, R, C, dtype, s);
        if (rc == SDFG_OK) rc = run_pass_sequence(a, b, a, ks, R, C, ldp, dtype, c, st, s, &fin);
        if (rc == SDFG_OK) rc = launch_copy2d(out, ld, fin, ldp, R, C, dtype, s);
        scratch_free(a, s);
        scratch_free(b, s);
        return rc;
    }
    if (in_disposable && in != out) {
        void *fin = nullptr;
        rc = run_pass_sequence(in, out, const_cast<void *>(in), ks, R, C, ld, dtype, c, st, s, &fin);
        if (rc == SDFG_OK && fin != out) rc = launch_copy2d(out, ld, fin, ld, R, C, dtype, s);
        return rc;
    }
    void *scr = nullptr;
    rc = scratch_alloc(&scr, static_cast<size_t>(R) * ld * S, s);
    if (rc != SDFG_OK) return rc;
    void *first, *second;
    if (in != out) {
        first = (n_steps_total % 2 == 1) ? out : scr;
        second = (first == out) ? scr : out;
    } else {
        first = scr;
        second = out;
    }
    void *fin = nullptr;
    rc = run_pass_sequence(in, first, second, ks, R, C, ld, dtype, c, st, s, &fin);
    if (rc == SDFG_OK && fin != out) rc = launch_copy2d(out, ld, fin, ld, R, C, dtype, s);
    scratch_free(scr, s);
    return rc;
}

// Temporal (or naive) path with a scratch grid the caller provides (R x ld
// elements, not overlapping in/out); allocates nothing.  `st` may describe a
// device whose error word lives in caller-provided memory.
int run_single_with_scratch(const void *in, void *out, void *scratch, int R, int C, int ld, long long T, int dtype,
                            const sdfg_config *cfg, DeviceState *st, cudaStream_t s) {
    if (R == 0 || C == 0) return SDFG_OK;
    if (T == 0 || R < 3 || C < 3) return launch_copy2d(out, ld, in, ld, R, C, dtype, s);
    sdfg_config c;
    int rc = resolve_config(cfg, R, C, dtype, true, &c);
    if (rc != SDFG_OK) return rc;
    if (c.kernel != SDFG_KERNEL_NAIVE) c.kernel = SDFG_KERNEL_TEMPORAL;
    const std::vector<int> ks = c.kernel == SDFG_KERNEL_NAIVE ? std::vector<int>(1, static_cast<int>(T))
                                                              : plan_passes(T, c.k);
    const long long n_steps_total = c.kernel == SDFG_KERNEL_NAIVE ? T : static_cast<long long>(ks.size());
    void *first, *second;
    if (in != out) {
        first = (n_steps_total % 2 == 1) ? out : scratch;
        second = (first == out) ? scratch : out;
    } else {
        first = scratch;
        second = out;
    }
    void *fin = nullptr;
    rc = run_pass_sequence(in, first, second, ks, R, C, ld, dtype, c, st, s, &fin);
    if (rc == SDFG_OK && fin != out) rc = launch_copy2d(out, ld, fin, ld, R, C, dtype, s);
    return rc;
}

}  // namespace sdfg

using namespace sdfg;

extern "C" int sdfg_jacobi2d_cfg(const void *in, void *out, int rows, int cols, int ld, int T, int dtype,
                                 const sdfg_config *cfg, void *stream) {
    int rc = validate_grid(in, out, rows, cols, ld, T, dtype, "sdfg_jacobi2d");
    if (rc != SDFG_OK) return rc;
    return run_single(in, out, rows, cols, ld, T, dtype, cfg, false, static_cast<cudaStream_t>(stream));
}

extern "C" int sdfg_jacobi2d_ex(const void *in, void *out, int rows, int cols, int ld, int T, int dtype,
                                void *stream) {
    return sdfg_jacobi2d_cfg(in, out, rows, cols, ld, T, dtype, nullptr, stream);
}

extern "C" int sdfg_jacobi2d(const float *in, float *out, int rows, int cols, int T, void *stream) {
    return sdfg_jacobi2d_cfg(in, out, rows, cols, cols, T, SDFG_F32, nullptr, stream);
}

namespace {
// Device buffers reused by sdfg_jacobi2d_host between calls of the same size.
struct HostCallCache {
    std::mutex mu;
    int device = -1;
    size_t bytes = 0;
    void *a = nullptr, *b = nullptr;
};
HostCallCache g_host_cache;
}  // namespace

extern "C" int sdfg_jacobi2d_host(const void *h_in, void *h_out, int rows, int cols, int T, int dtype,
                                  void *stream) {
    int rc = validate_grid(h_in, h_out, rows, cols, cols, T, dtype, "sdfg_jacobi2d_host");
    if (rc != SDFG_OK) return rc;
    if (rows == 0 || cols == 0) return SDFG_OK;
    DeviceState *st = nullptr;
    rc = current_device(&st);
    if (rc != SDFG_OK) return rc;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const size_t bytes = static_cast<size_t>(rows) * cols * dtype_bytes(dtype);
    std::lock_guard<std::mutex> lk(g_host_cache.mu);
    if (g_host_cache.device != st->device || g_host_cache.bytes < bytes) {
        if (g_host_cache.a) cudaFree(g_host_cache.a);
        if (g_host_cache.b) cudaFree(g_host_cache.b);
        g_host_cache.a = g_host_cache.b = nullptr;
        g_host_cache.bytes = 0;
        SDFG_CUDA(cudaMalloc(&g_host_cache.a, bytes));
        SDFG_CUDA(cudaMalloc(&g_host_cache.b, bytes));
        g_host_cache.bytes = bytes;
        g_host_cache.device = st->device;
    }
    TimedLaunch t_in = stats_begin(FAM_H2D, s);
    cudaError_t e = cudaMemcpyAsync(g_host_cache.a, h_in, bytes, cudaMemcpyHostToDevice, s);
    stats_end(t_in, s);
    if (e != cudaSuccess) return cuda_error(e, "cudaMemcpyAsync (host to device)");
    rc = run_single(g_host_cache.a, g_host_cache.b, rows, cols, cols, T, dtype, nullptr, true, s);
    if (rc != SDFG_OK) return rc;
    TimedLaunch t_out = stats_begin(FAM_D2H, s);
    e = cudaMemcpyAsync(h_out, g_host_cache.b, bytes, cudaMemcpyDeviceToHost, s);
    stats_end(t_out, s);
    if (e != cudaSuccess) return cuda_error(e, "cudaMemcpyAsync (device to host)");
    SDFG_CUDA(cudaStreamSynchronize(s));
    return SDFG_OK;
}

namespace {
// Two device slots (input, result) and two streams for sdfg_jacobi2d_host_many.
struct HostPipe {
    std::mutex mu;
    int device = -1;
    size_t bytes = 0;
    void *in[2] = {nullptr, nullptr}, *out[2] = {nullptr, nullptr};
    cudaStream_t q[2] = {nullptr, nullptr};
    cudaEvent_t ev[3] = {nullptr, nullptr, nullptr};  // caller ready, slot 0 done, slot 1 done
};
constexpr int kHostPipeDevices = 64;
HostPipe g_host_pipe[kHostPipeDevices];  // one pair of slots per device

int host_pipe_ready(HostPipe &hp, int device, size_t bytes) {
    if (!hp.q[0]) {
        for (int i = 0; i < 2; ++i) SDFG_CUDA(cudaStreamCreateWithFlags(&hp.q[i], cudaStreamNonBlocking));
        for (int i = 0; i < 3; ++i) SDFG_CUDA(cudaEventCreateWithFlags(&hp.ev[i], cudaEventDisableTiming));
        hp.device = device;
    }
    if (hp.bytes < bytes) {
        SDFG_CUDA(cudaDeviceSynchronize());  // the slots may still be in use by the streams
        for (int i = 0; i < 2; ++i) {
            if (hp.in[i]) cudaFree(hp.in[i]);
            if (hp.out[i]) cudaFree(hp.out[i]);
            hp.in[i] = hp.out[i] = nullptr;
        }
        hp.bytes = 0;
        for (int i = 0; i < 2; ++i) {
            SDFG_CUDA(cudaMalloc(&hp.in[i], bytes));
            SDFG_CUDA(cudaMalloc(&hp.out[i], bytes));
        }
        hp.bytes = bytes;
    }
    return SDFG_OK;
}
}  // namespace

// n independent solves of host grids, pipelined: solve i runs on slot i % 2
// (its own device input and result buffers, its own stream), so the copies
// of one solve overlap the computation of the next.  Same operation and
// results as n calls of sdfg_jacobi2d_host.
extern "C" int sdfg_jacobi2d_host_many(const void *const *h_in, void *const *h_out, int n, int rows, int cols, int T,
                                       int dtype, void *stream) {
    if (n < 0 || (n > 0 && (!h_in || !h_out)))
        return set_error(SDFG_ERR_INVAL, "sdfg_jacobi2d_host_many: n=%d with null arrays", n);
    for (int i = 0; i < n; ++i) {
        int rc = validate_grid(h_in[i], h_out[i], rows, cols, cols, T, dtype, "sdfg_jacobi2d_host_many");
        if (rc != SDFG_OK) return rc;
    }
    if (n == 0 || rows == 0 || cols == 0) return SDFG_OK;
    DeviceState *st = nullptr;
    int rc = current_device(&st);
    if (rc != SDFG_OK) return rc;
    if (st->device < 0 || st->device >= kHostPipeDevices)
        return set_error(SDFG_ERR_UNSUPPORTED, "sdfg_jacobi2d_host_many: device %d", st->device);
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const size_t bytes = static_cast<size_t>(rows) * cols * dtype_bytes(dtype);
    HostPipe &hp = g_host_pipe[st->device];
    std::lock_guard<std::mutex> lk(hp.mu);
    rc = host_pipe_ready(hp, st->device, bytes);
    if (rc != SDFG_OK) return rc;
    // on a failure after work was queued, let that work finish (its copies
    // read and write the caller's host buffers) before returning
    auto fail = [&](int code) {
        for (int q = 0; q < 2; ++q) cudaStreamSynchronize(hp.q[q]);
        return code;
    };
    // both slot streams start after the work already on the caller's stream
    SDFG_CUDA(cudaEventRecord(hp.ev[0], s));
    for (int q = 0; q < 2; ++q) SDFG_CUDA(cudaStreamWaitEvent(hp.q[q], hp.ev[0], 0));
    for (int i = 0; i < n; ++i) {
        const int q = i & 1;
        cudaStream_t qs = hp.q[q];
        TimedLaunch t_in = stats_begin(FAM_H2D, qs);
        cudaError_t e = cudaMemcpyAsync(hp.in[q], h_in[i], bytes, cudaMemcpyHostToDevice, qs);
        stats_end(t_in, qs);
        if (e != cudaSuccess) return fail(cuda_error(e, "cudaMemcpyAsync (host to device)"));
        rc = run_single(hp.in[q], hp.out[q], rows, cols, cols, T, dtype, nullptr, true, qs);
        if (rc != SDFG_OK) return fail(rc);
        TimedLaunch t_out = stats_begin(FAM_D2H, qs);
        e = cudaMemcpyAsync(h_out[i], hp.out[q], bytes, cudaMemcpyDeviceToHost, qs);
        stats_end(t_out, qs);
        if (e != cudaSuccess) return fail(cuda_error(e, "cudaMemcpyAsync (device to host)"));
    }
    // the caller's stream resumes after both slots; return when every h_out holds its result
    for (int q = 0; q < 2; ++q) {
        cudaError_t e = cudaEventRecord(hp.ev[1 + q], hp.q[q]);
        if (e == cudaSuccess) e = cudaStreamWaitEvent(s, hp.ev[1 + q], 0);
        if (e != cudaSuccess) return fail(cuda_error(e, "sdfg_jacobi2d_host_many: stream order"));
    }
    SDFG_CUDA(cudaStreamSynchronize(s));
    return SDFG_OK;
}
