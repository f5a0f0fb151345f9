// Halo exchange between the CTAs of one cooperative launch through words in
// global memory (tiles.cuh, tiles64.cu).
#pragma once

#include "device_common.cuh"

namespace sdfg {

constexpr uint32_t LL_NEVER = 1u << 31;  // added to a pass's number: one that no launch reaches

// Exchange words: a value and the number of the pass it belongs to in one
// 64-bit word, two words per 16-byte access.  A word arrives whole, so the
// reader needs no flag and no fence: it reads until every word bears the pass
// it waits for.  (Data and flag in one word is the idea of the low-latency
// protocol, LL, of NVIDIA's NCCL, whose public documents describe it.)
__device__ __forceinline__ void ll_store(uint64_t *p, float x, float y, uint32_t pass) {
    asm volatile(
        "{\n\t.reg .b64 a, b;\n\t"
        "mov.b64 a, {%1, %3};\n\t"
        "mov.b64 b, {%2, %3};\n\t"
        "st.relaxed.gpu.global.v2.b64 [%0], {a, b};\n\t}" ::"l"(p),
        "r"(__float_as_uint(x)), "r"(__float_as_uint(y)), "r"(pass)
        : "memory");
}
__device__ __forceinline__ bool ll_load(float &x, float &y, const uint64_t *p, uint32_t pass) {
    uint32_t vx, vy, ex, ey;
    asm volatile(
        "{\n\t.reg .b64 a, b;\n\t"
        "ld.relaxed.gpu.global.v2.b64 {a, b}, [%4];\n\t"
        "mov.b64 {%0, %2}, a;\n\t"
        "mov.b64 {%1, %3}, b;\n\t}"
        : "=r"(vx), "=r"(vy), "=r"(ex), "=r"(ey)
        : "l"(p)
        : "memory");
    x = __uint_as_float(vx);
    y = __uint_as_float(vy);
    return ex == pass && ey == pass;
}

// A value of 64 bits as two words.
__device__ __forceinline__ void ll_store(uint64_t *p, double x, uint32_t pass) {
    ll_store(p, __int_as_float(__double2loint(x)), __int_as_float(__double2hiint(x)), pass);
}
__device__ __forceinline__ bool ll_load(double &x, const uint64_t *p, uint32_t pass) {
    float lo, hi;
    const bool ok = ll_load(lo, hi, p, pass);
    x = __hiloint2double(__float_as_int(hi), __float_as_int(lo));
    return ok;
}

// Bounded waits of one warp.
struct LLWait {
    unsigned long long timeout_ns;
    int *err;
    bool dead;  // a wait ran out: the error word is set, no further wait
    // Repeats `attempt` (all lanes' loads) until every lane has what it waits for.
    template <class Attempt> __device__ __forceinline__ void until(Attempt attempt) {
        if (dead) return;
        unsigned long long t0 = 0;
        for (int n = 1; !__all_sync(FULL_MASK, attempt()); ++n) {
            if (n % 64) continue;
            const unsigned long long t = globaltimer_ns();
            if (t0 == 0) t0 = t;
            if (__any_sync(FULL_MASK, t - t0 > timeout_ns)) {
                dead = true;
                if ((threadIdx.x & 31) == 0) set_device_error(err, DEV_ERR_TIMEOUT_DEP);
                return;
            }
        }
    }
};

}  // namespace sdfg
