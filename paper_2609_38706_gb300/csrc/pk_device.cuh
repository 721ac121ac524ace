// pk_device.cuh -- small device helpers shared by the libpk kernels.
#pragma once
#include <stdint.h>

#include "../../include/pk.h"

namespace pk {

__device__ __forceinline__ void set_status(int32_t *status, int32_t code) {
    if (status) atomicCAS(status, 0, code);
}

// Request index r with key_off[r] <= g < key_off[r+1], for a non-decreasing
// key_off with key_off[0] <= g < key_off[R].  Called by all 32 lanes of a warp
// with the same g: each level probes 32 positions at once, so R = 2^14
// requests resolve in 3 rounds of independent loads instead of 14 dependent
// ones.
__device__ __forceinline__ uint32_t warp_find_request(const int64_t *key_off, uint32_t R,
                                                      int64_t g) {
    const uint32_t lane = threadIdx.x & 31;
    uint32_t lo = 0, hi = R;  // key_off[lo] <= g < key_off[hi]
    while (hi - lo > 1) {
        const uint32_t span = hi - lo;
        const uint32_t step = span > 32 ? span / 32 : 1;  // span <= 32: every candidate probed at once
        uint32_t p = lo + (lane + 1) * step;
        if (p > hi - 1) p = hi - 1;
        const bool le = __ldcg(key_off + p) <= g;
        const uint32_t ball = __ballot_sync(0xffffffffu, le);
        // probes are non-decreasing in lane, so the set lanes form a prefix
        const int last = 31 - __clz(ball);  // -1 if none
        const uint32_t new_lo = last >= 0 ? __shfl_sync(0xffffffffu, p, last) : lo;
        const int next = last + 1;
        const uint32_t new_hi = next <= 31 ? __shfl_sync(0xffffffffu, p, next) : hi;
        lo = new_lo;
        hi = (new_hi > lo) ? new_hi : hi;
        if (span <= 32) break;
    }
    return lo;
}

// Same, for one thread, restricted to [lo, hi) known to contain the answer.
__device__ __forceinline__ uint32_t find_request_in(const int64_t *key_off, uint32_t lo, uint32_t hi,
                                                    int64_t g) {
    while (hi - lo > 1) {
        const uint32_t mid = (lo + hi) >> 1;
        if (__ldcg(key_off + mid) <= g) lo = mid; else hi = mid;
    }
    return lo;
}

// Per-lane request of item g (items of one warp are g0 .. g0+31, g0 the
// warp's first item, all lanes active).  `total` = key_off[R].
__device__ __forceinline__ uint32_t lane_request(const int64_t *key_off, uint32_t R, int64_t g0,
                                                 int64_t total, int64_t g) {
    const uint32_t r0 = warp_find_request(key_off, R, g0);
    int64_t g_last = g0 + 31;
    if (g_last >= total) g_last = total - 1;
    const uint32_t r1 = warp_find_request(key_off, R, g_last);
    return find_request_in(key_off, r0, r1 + 1, g < total ? g : total - 1);
}

// Same result as lane_request, in code whose control flow is uniform over the
// warp as far as the compiler can see: every branch is on a vote and every loop
// runs a number of times that follows from R alone.  A loop or branch that may
// diverge, even one that never runs, costs the code after it the uniform data
// path (the chunk digests of batches of equal requests, whose mapping never
// left its first lines: with divergent searches in the fallback and a divergent
// end of the batch, sweep key derivation 207 us, small-block 613.8; 196.5 and
// 591.9 so).
//
// First a guess for batches of about equal requests, r_g = g0 * R / total, and
// one 32-wide load of key_off[w0 ..], w0 = r_g - 8.  With p_j = key_off[w0 + j] -
// g0 clamped to 0..32, item g0 + l lies in request w0 + (number of p_j <= l) - 1:
// the p_j = 0 by a ballot, the others by a mask of their positions when they
// differ (no empty requests among them).  When the window does not bracket the
// warp's items, or requests in it are empty: a 32-ary search for the request r0
// of the first item, the same window from r0 counted by a search over shuffles,
// and for items past those 32 requests (after runs of empty ones) a binary
// search of key_off.
__device__ __forceinline__ uint32_t lane_request_guess(const int64_t *key_off, uint32_t R, int64_t g0,
                                                       int64_t total, int64_t g) {
    constexpr uint32_t kFull = 0xffffffffu;
    const uint32_t lane = threadIdx.x & 31;
    const int64_t gg = g < total ? g : total - 1;
    const uint32_t l = (uint32_t)(gg - g0);  // this lane's item, 0..31
    auto window = [&](uint32_t w0) {         // p of key_off[w0 + lane]
        const uint64_t at = (uint64_t)w0 + lane;
        const int64_t d = (at <= R ? __ldcg(key_off + at) : INT64_MAX) - g0;
        return d <= 0 ? 0u : d > 31 ? 32u : (uint32_t)d;
    };
    const uint32_t last = total - g0 < 32 ? (uint32_t)(total - g0) - 1 : 31u;
    uint32_t rg = (uint32_t)((float)g0 / (float)total * (float)R);
    rg = rg >= R ? R - 1 : rg;
    const uint32_t w0 = rg > 8 ? rg - 8 : 0;
    uint32_t p = window(w0);
    const uint32_t before = __ballot_sync(kFull, p == 0), among = __ballot_sync(kFull, p - 1 < 31);
    const uint32_t places = __reduce_or_sync(kFull, p - 1 < 31 ? 1u << p : 0u);
    if ((before & 1u) && __ballot_sync(kFull, p > last) && __popc(places) == __popc(among))
        return w0 + __popc(before) - 1 + __popc(places & ((2u << l) - 1u));
    // the request r0 of item g0: blocks of `step` requests, the last one that starts at or before g0
    uint32_t r0 = 0;
    for (uint32_t span = R; span > 1;) {
        const uint32_t step = (span + 31) / 32;
        const uint64_t c = (uint64_t)r0 + (uint64_t)(lane + 1) * step;
        r0 += step * __popc(__ballot_sync(kFull, c < R && __ldcg(key_off + c) <= g0));
        span = step;
    }
    // items within the 32 requests from r0: the number of boundaries among key_off[r0 + 1 ..] at or before the item
    p = window(r0 + 1);
    uint32_t lo = 0, hi = 32;
#pragma unroll 1
    for (int it = 0; it < 6; ++it) {
        const uint32_t mid = (lo + hi) >> 1;
        const uint32_t pm = __shfl_sync(kFull, p, mid < 31 ? mid : 31);
        const bool up = lo < hi && pm <= l;
        hi = lo < hi && !up ? mid : hi;
        lo = up ? mid + 1 : lo;
    }
    if (__all_sync(kFull, lo < 32)) return r0 + lo;
    uint32_t r = r0;
#pragma unroll 1
    for (uint32_t n = R - r0; n > 1;) {  // the last request of the n from r that starts at or before the item
        const uint32_t h = n >> 1;
        r = __ldcg(key_off + r + h) <= gg ? r + h : r;
        n -= h;
    }
    return r;
}

}  // namespace pk

namespace pk {

// Programmatic dependent launch (sm_90+).  Every libpk kernel is launched with
// programmatic stream serialization: it may become resident while the previous
// kernel of the stream drains, and waits for its predecessor's completion (and
// memory) before touching global memory.  Kernels release their successor
// once their main work is done (short kernels at their start): a successor
// released early sits on the SMs, with its own successor, for the whole run of
// the kernel (multi-adapter batch: key derivation 82 -> 74 us, small-block
// step 1073 -> 909 us when the digest and chain kernels release late).  Both
// are no-ops for a kernel launched without the attribute.
//
// Memory written by a predecessor is read only with coherent loads (plain or
// L2 loads: __ldcg, ld.global.cg), never through the non-coherent read-only
// path (__ldg, ld.global.nc, loads through const __restrict__ pointers): a
// kernel resident while its predecessor still writes can read stale data on
// that path even after the wait (measured: a store in range mode reading the
// lookup's h_r as 0).  pdl_wait(p...) also passes the kernel's pointers
// through an empty asm after the wait, so that no access through them is
// scheduled before it.
template <typename P>
__device__ __forceinline__ void launder(P &p) {
    asm volatile("" : "+l"(p));
}
template <typename... P>
__device__ __forceinline__ void pdl_wait(P &...p) {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    (launder(p), ...);
}
__device__ __forceinline__ void pdl_launch_dependents() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

}  // namespace pk
