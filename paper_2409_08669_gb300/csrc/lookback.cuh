// Decoupled lookback over the run counts of the depth-ordered Gaussians, shared
// by the run scan (emit.cu) and the window sort that carries its own scan
// (bins.cu).
#pragma once

#include "adr_internal.cuh"

namespace adr {

constexpr uint32_t kSat = 0x7FFFFFFFu;   // running sums saturate here (> any capacity)
constexpr unsigned long long kScanInc = 1ull << 31;

__device__ __forceinline__ uint32_t sat_add(uint32_t a, uint32_t b) {
    const uint32_t s = a + b;
    return (s < a || s > kSat) ? kSat : s;
}

// Exclusive prefix of chunk `chunk` by decoupled lookback, run by one warp:
// lane l reads the word of chunk j - l, so each round trip covers 32
// predecessors; the words up to the nearest inclusive prefix are summed.
// Lane 0 publishes this chunk's aggregate first and its inclusive prefix last
// (except the chunk the testing hook withholds).  A wait that makes no
// progress for lt.spin_limit polls gives up: it flags the status word, sets
// *gave_up and returns the partial prefix.
__device__ __forceinline__ uint32_t warp_lookback(unsigned long long* lookback, uint32_t chunk, uint32_t total,
                                  uint32_t epoch, uint32_t* status, LookbackTest lt,
                                  bool* gave_up) {
    *gave_up = false;
    const int lane = threadIdx.x & 31;
    const unsigned long long tag = (unsigned long long)epoch << 32;
    volatile unsigned long long* lb = lookback;
    const bool publish = chunk != lt.withhold;
    if (chunk == 0) {
        if (lane == 0 && publish) lb[0] = tag | kScanInc | min(total, kSat);
        return 0;
    }
    if (lane == 0 && publish) lb[chunk] = tag | min(total, kSat);
    uint64_t excl = 0;
    int64_t j = (int64_t)chunk - 1;   // the nearest predecessor not yet summed
    int spins = 0;
    for (;;) {
        const int64_t idx = j - lane;
        // Before chunk 0 reads as an inclusive prefix of 0 (never reached:
        // chunk 0 always publishes one).
        const unsigned long long w = idx >= 0 ? lb[idx] : (tag | kScanInc);
        const bool ready = (uint32_t)(w >> 32) == epoch;
        const uint32_t not_ready = __ballot_sync(0xffffffffu, !ready);
        const uint32_t inc = __ballot_sync(0xffffffffu, ready && (w & kScanInc));
        const int first_nr = not_ready ? __ffs(not_ready) - 1 : 32;
        const int first_inc = inc ? __ffs(inc) - 1 : 32;
        const int take = first_inc < first_nr ? first_inc + 1 : first_nr;   // summed lanes
        uint64_t v = lane < take ? (uint64_t)((uint32_t)w & kSat) : 0ull;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        excl += v;
        if (first_inc < first_nr) break;
        j -= take;
        if (take == 0) {
            if (++spins > lt.spin_limit) {
                if (lane == 0) atomicOr(status, kErrLookback);
                *gave_up = true;
                break;
            }
            __nanosleep(32);
        }
    }
    const uint32_t e = (uint32_t)min(excl, (uint64_t)kSat);
    __threadfence();
    if (lane == 0 && publish) lb[chunk] = tag | kScanInc | sat_add(e, total);
    return e;
}

// The run chunks (of kMarkRuns runs) that start inside the runs [run, run + t)
// of the Gaussian at depth-order position i: each one's holder is i.
__device__ __forceinline__ void mark_chunks(uint32_t run, uint32_t t, uint32_t i, int64_t capacity,
                                            uint32_t* __restrict__ chunk_first) {
    // run < 2^31 and t <= 256, so run + t does not wrap
    uint32_t c = (run + (uint32_t)kMarkRuns - 1u) / (uint32_t)kMarkRuns;
    if (t == 0u || c * (uint32_t)kMarkRuns >= run + t || (int64_t)run >= capacity) return;
    const uint32_t c_max = (uint32_t)((capacity - 1) / kMarkRuns);
    for (; c * (uint32_t)kMarkRuns < run + t && c <= c_max; ++c) chunk_first[c] = i;
}

}  // namespace adr
