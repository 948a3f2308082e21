// Decoupled look-back (single-pass prefix over CTAs in ticket order).
// Each tile publishes its aggregate, then walks back over its predecessors
// until it meets an inclusive prefix, and publishes its own inclusive prefix.
// Every wait is bounded by a device-clock limit (limit_ns); on expiry the
// caller's timeout flag is set and the tile publishes its partial prefix
// marked as poisoned.  A tile that meets a poisoned prefix sets its own
// timeout flag and passes the poison on, so every tile after an expired wait
// reports it and no tile takes a partial prefix for a final one.
#pragma once
#include "pivco_dev.cuh"

namespace pv {

constexpr uint64_t kLbFlagAgg = 1ull << 62;
constexpr uint64_t kLbFlagInc = 2ull << 62;
constexpr uint64_t kLbPoison = 1ull << 61;
constexpr uint64_t kLbValMask = (1ull << 61) - 1;

__device__ inline void lb_store(uint64_t *p, uint64_t v) {
    asm volatile("st.release.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}
__device__ inline uint64_t lb_load(const uint64_t *p) {
    uint64_t v;
    asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}

// Called by ONE thread.  Returns the exclusive prefix of `agg` over tiles
// 0 .. tile-1.  states[] must be zero before the launch.
__device__ inline uint64_t lookback_exclusive(uint64_t *states, int tile, uint64_t agg, int *timed_out,
                                              uint64_t limit_ns) {
    if (tile == 0) {
        lb_store(&states[0], kLbFlagInc | (agg & kLbValMask));
        return 0;
    }
    lb_store(&states[tile], kLbFlagAgg | (agg & kLbValMask));
    uint64_t excl = 0;
    int j = tile - 1;
    bool bad = false;
    const uint64_t t0 = globaltimer_ns();
    unsigned ns = 32;
    while (j >= 0) {
        const uint64_t v = lb_load(&states[j]);
        const uint64_t f = v & (kLbFlagAgg | kLbFlagInc);
        if (f == 0) {
            if (globaltimer_ns() - t0 > limit_ns) { bad = true; break; }
            __nanosleep(ns);
            if (ns < 1024) ns <<= 1;
            continue;
        }
        excl += v & kLbValMask;
        if (f == kLbFlagInc) {
            bad = (v & kLbPoison) != 0;
            break;
        }
        j--;
    }
    if (bad) *timed_out = 1;
    lb_store(&states[tile], kLbFlagInc | (bad ? kLbPoison : 0ull) | ((excl + agg) & kLbValMask));
    return excl;
}

// Two chains walked by a whole CTA (kLbThreads threads): each step reads the
// states of the kLbThreads predecessors below j at once, so a first wave of
// CTAs that have all published only their aggregates is crossed in two or
// three round trips to L2 (a warp's 16 predecessors a step take forty).
// lb2_publish (one thread) makes the tile's own aggregates visible, before
// the tile's other work; lookback2_cta waits for the predecessors' (bounded),
// publishes the inclusive prefixes and returns the exclusive ones in every
// thread.  Returns true when the wait ran out or a poisoned prefix was met.
// A state holds all that is taken from it, so its loads and stores order
// nothing else (as acquire loads and release stores, 512 loads a CTA: batched,
// 600 blocks of 4096 symbols decoded in 58 us, 64 of 3000 in 43; now 51 and 35).
constexpr int kLbThreads = 256;
constexpr int kLbWarps = kLbThreads / 32;
__device__ inline void lb2_store(uint64_t *p, uint64_t v) {
    asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}
__device__ inline uint64_t lb2_load(const uint64_t *p) {
    uint64_t v;
    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}
__device__ inline void lb2_publish(uint64_t *states_a, uint64_t *states_b, int tile, uint64_t agg_a, uint64_t agg_b) {
    const uint64_t f = tile == 0 ? kLbFlagInc : kLbFlagAgg;
    lb2_store(&states_a[tile], f | (agg_a & kLbValMask));
    lb2_store(&states_b[tile], f | (agg_b & kLbValMask));
}
__device__ inline bool lookback2_cta(uint64_t *states_a, uint64_t *states_b, int tile, uint64_t agg_a, uint64_t agg_b,
                                     uint64_t &excl_a, uint64_t &excl_b, uint64_t limit_ns, uint32_t (*mins)[4],
                                     uint64_t (*sums)[2]) {
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    excl_a = excl_b = 0;
    if (tile == 0) return false;
    int j = tile - 1;
    bool bad = false;
    const uint64_t t0 = globaltimer_ns();
    unsigned ns = 32;
    for (;;) {
        const int k = j - t;
        const uint64_t va = k >= 0 ? lb2_load(&states_a[k]) : kLbFlagInc;   // before tile 0: an inclusive zero
        const uint64_t vb = k >= 0 ? lb2_load(&states_b[k]) : kLbFlagInc;
        const uint64_t fa = va & (kLbFlagAgg | kLbFlagInc), fb = vb & (kLbFlagAgg | kLbFlagInc);
        // both chains are published one right after the other: a state counts once they agree
        const bool inc = fa == kLbFlagInc && fb == kLbFlagInc, agg = fa == kLbFlagAgg && fb == kLbFlagAgg;
        const uint32_t mi = __reduce_min_sync(0xffffffffu, inc ? (uint32_t)t : (uint32_t)kLbThreads);
        const uint32_t mu = __reduce_min_sync(0xffffffffu, inc || agg ? (uint32_t)kLbThreads : (uint32_t)t);
        // (one thread's clock decides for the CTA)
        if (lane == 0) {
            mins[warp][0] = mi;
            mins[warp][1] = mu;
            mins[warp][2] = t == 0 && globaltimer_ns() - t0 > limit_ns;
        }
        __syncthreads();
        uint32_t ti = kLbThreads, tu = kLbThreads;
#pragma unroll
        for (int w = 0; w < kLbWarps; w++) { ti = min(ti, mins[w][0]); tu = min(tu, mins[w][1]); }
        const bool expired = mins[0][2] != 0;
        const bool take = (uint32_t)t <= ti;   // up to the nearest inclusive prefix
        uint64_t xa = take ? va & kLbValMask : 0ull, xb = take ? vb & kLbValMask : 0ull;
#pragma unroll
        for (int o = 16; o; o >>= 1) {
            xa += __shfl_xor_sync(0xffffffffu, xa, o);
            xb += __shfl_xor_sync(0xffffffffu, xb, o);
        }
        const bool pois = (uint32_t)t == ti && ((va | vb) & kLbPoison) != 0;
        if (lane == 0) { sums[warp][0] = xa; sums[warp][1] = xb; }
        const bool anyp = __syncthreads_or(pois) != 0;
        if (tu < ti) {   // a state needed is not there yet
            if (expired) { bad = true; break; }
            __nanosleep(ns);
            if (ns < 512) ns <<= 1;
            __syncthreads();
            continue;
        }
#pragma unroll
        for (int w = 0; w < kLbWarps; w++) { excl_a += sums[w][0]; excl_b += sums[w][1]; }
        if (ti < (uint32_t)kLbThreads) { bad = anyp; break; }
        j -= kLbThreads;
        __syncthreads();
    }
    __syncthreads();
    if (t == 0) {
        const uint64_t p = bad ? kLbPoison : 0ull;
        lb2_store(&states_a[tile], kLbFlagInc | p | ((excl_a + agg_a) & kLbValMask));
        lb2_store(&states_b[tile], kLbFlagInc | p | ((excl_b + agg_b) & kLbValMask));
    }
    return bad;
}

}  // namespace pv
