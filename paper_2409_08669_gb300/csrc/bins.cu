// The view-depth order of the Gaussians with tiles (the depth half of the
// paper's (tile | depth) sort key, Sec. 3.2.1) by binning, with stage 2, the
// scan of their column runs, in its last kernel.
//
// Preprocess adds every kept Gaussian to a histogram of its depth key (the
// key's distance from the nearest key in units of 2^shift; a depth octave is
// 512 to 8192 bins, by the scene's size) and keeps the count it found there,
// its arrival rank in the bin.  Then
//   k_bin_scan     turns the histogram into every bin's start (one cluster of 8
//                  CTAs, block totals exchanged through distributed shared
//                  memory) and finds where the windows begin: window w holds
//                  the bins that start at positions [w kWindow, (w + 1) kWindow);
//   k_bin_scatter  writes each Gaussian's (key, index) at its bin's start plus
//                  its rank: the Gaussians are grouped by bin, in no order inside;
//   k_window_sort  sorts one window at a time on chip and scans its run counts.
// Keys equal in all 32 bits are ordered by Gaussian index, so the result is
// that of the stable radix sort (sort.cu), whatever order the arrivals took.
//
// The radix sort's four passes are twelve launches whose time is the latency
// of one 4096-key chunk's chain (load, sixteen ranking rounds, prefix,
// write-out) several times over, whatever the number of keys; here a key is
// moved once through memory and once through shared memory.  With the run scan
// that both need: 88 us by the passes at 10k Gaussians (of a 155 us frame) and 100 at
// 1M, 21 and 25 us by these three kernels (at 1M of depth slice 0), each 5 to 10 us
// of latency.
#include <cooperative_groups.h>

#include "lookback.cuh"

namespace adr {
namespace {

namespace cg = cooperative_groups;

constexpr int kScanCluster = 8;          // CTAs of k_bin_scan
constexpr int kWinThreads = 256;
constexpr int kWinItems = 8;
constexpr int kWinCap = kWinThreads * kWinItems;   // Gaussians of a window sorted on chip
constexpr int kLargeItems = 4;           // per thread and round of the large windows' radix sort
constexpr int kSubBits = 12;
constexpr int kSub = 1 << kSubBits;      // sub-bins of a window's key range
constexpr int kWinWarps = kWinThreads / 32;
// Most members of a sub-bin that are placed by comparing each with all: 8 a thread at 20 ns each are 20 us,
// what the radix sort of a window takes (2000 Gaussians at one depth, whole frame: 438 us -> 81).
constexpr uint32_t kCrowded = 128;

// ---------------------------------------------------------------------------
// Bin starts and window starts.  Warp w of CTA r holds the 128 kQuads bins from
// 128 kQuads (r * warps + w) on, 4 consecutive bins a lane and load.
// ---------------------------------------------------------------------------
template <int kQuads>
__global__ void __cluster_dims__(kScanCluster, 1, 1)
k_bin_scan(uint32_t* __restrict__ bins, uint32_t* __restrict__ win_lo, int what, uint32_t* __restrict__ counters,
           uint32_t* __restrict__ slices, const unsigned long long* __restrict__ sums, int64_t capacity,
           uint32_t* __restrict__ largest, uint32_t* __restrict__ status) {
    pdl_prologue();
    __shared__ uint32_t s_w[32], s_max[32];
    __shared__ uint32_t s_total, s_cta_max;
    cg::cluster_group cluster = cg::this_cluster();
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, warps = (int)blockDim.x >> 5;
    const uint32_t rank = cluster.block_rank();
    uint4* b4 = reinterpret_cast<uint4*>(bins) + (size_t)(rank * (uint32_t)warps + (uint32_t)warp) * 32 * kQuads + lane;
    uint4 v[kQuads];
    uint32_t first[kQuads], sum = 0, big = 0;   // first: the warp's items before this lane's quad
#pragma unroll
    for (int q = 0; q < kQuads; ++q) v[q] = b4[32 * q];
#pragma unroll
    for (int q = 0; q < kQuads; ++q) {
        const uint32_t t = v[q].x + v[q].y + v[q].z + v[q].w;
        big = max(big, max(max(v[q].x, v[q].y), max(v[q].z, v[q].w)));
        uint32_t incl = t;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += y;
        }
        first[q] = sum + incl - t;
        sum += __shfl_sync(0xffffffffu, incl, 31);
    }
    big = __reduce_max_sync(0xffffffffu, big);
    if (lane == 0) {
        s_w[warp] = sum;
        s_max[warp] = big;
    }
    __syncthreads();
    uint32_t before = 0;
    for (int w = 0; w < warp; ++w) before += s_w[w];
    if (tid == (int)blockDim.x - 1) {
        s_total = before + sum;
        uint32_t m = 0;
        for (int w = 0; w < warps; ++w) m = max(m, s_max[w]);
        s_cta_max = m;
    }
    cluster.sync();
    uint32_t total = 0, most = 0;
#pragma unroll
    for (uint32_t r = 0; r < (uint32_t)kScanCluster; ++r) {
        const uint32_t t = *cluster.map_shared_rank(&s_total, r);
        most = max(most, *cluster.map_shared_rank(&s_cta_max, r));
        before += r < rank ? t : 0u;
        total += t;
    }
    // A bin [s, e): the windows it starts (s a multiple of kWindow) begin at s;
    // the windows whose first position falls inside it begin at e.  Depth slice 0
    // ends with the bin that holds its last Gaussian.
    const uint32_t K0 = what == kScanFrame ? slice0_count(total) : 0u;
    auto place = [&](uint32_t s, uint32_t& c, uint32_t bin) {
        const uint32_t e = s + c;
        if (c != 0u) {
            uint32_t w = (s + (uint32_t)kWindow - 1u) / (uint32_t)kWindow;
            if (w * (uint32_t)kWindow == s) win_lo[w++] = s;
            for (; w * (uint32_t)kWindow < e; ++w) win_lo[w] = e;
            if (s < K0 && K0 <= e) {
                counters[kCntSliceBin] = bin + 1u;
                if (slices) slices[kCntVisible] = slices[kCntDepthKept] = e;
            }
        }
        c = s;
        return e;
    };
    auto crosses = [&](uint32_t s, uint32_t e) {   // a window begins in [s, e), or slice 0 ends in (s, e]
        return (s + (uint32_t)kWindow - 1u) / (uint32_t)kWindow != (e + (uint32_t)kWindow - 1u) / (uint32_t)kWindow ||
               (s < K0 && K0 <= e);
    };
#pragma unroll
    for (int q = 0; q < kQuads; ++q) {
        uint32_t s = before + first[q];
        uint4 c = v[q];
        const uint32_t bin = (((rank * (uint32_t)warps + (uint32_t)warp) * kQuads + q) * 32u + (uint32_t)lane) * 4u;
        if (crosses(s, s + c.x + c.y + c.z + c.w)) {
            s = place(s, c.x, bin);
            s = place(s, c.y, bin + 1u);
            s = place(s, c.z, bin + 2u);
            place(s, c.w, bin + 3u);
        } else {
            c = make_uint4(s, s + c.x, s + c.x + c.y, s + c.x + c.y + c.z);
        }
        b4[32 * q] = c;
    }
    if (rank == 0 && warp == 0) {
        if (what == kScanFrame) {   // Preprocess's sums, saturated to 31 bits
            unsigned long long p = 0, r = 0;
            for (int k = lane; k < kSumSlots; k += 32) {
                p += sums[kSumStride * k];
                r += sums[kSumStride * k + 1];
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                p += __shfl_xor_sync(0xffffffffu, p, o);
                r += __shfl_xor_sync(0xffffffffu, r, o);
            }
            if (lane == 0) {
                const uint32_t pairs = (uint32_t)min(p, (unsigned long long)kSat);
                counters[kCntPairs] = pairs;
                counters[kCntRuns] = (uint32_t)min(r, (unsigned long long)kSat);
                counters[kCntVisible] = counters[kCntDepthKept] = total;
                if (slices) slices[kCntPairs] = pairs;
                if (p > (unsigned long long)capacity) atomicOr(status, kErrCapacity);
            }
        } else if (what == kScanSlice1 && lane == 0) {
            uint32_t* c1 = slices + kCntSlots;
            c1[kCntVisible] = c1[kCntDepthKept] = total;
            c1[kCntPairs] = counters[kCntPairs];
        }
        if (lane == 0) {
            win_lo[(total + (uint32_t)kWindow - 1u) / (uint32_t)kWindow] = total;
            if (what != kScanSlice1) {
                if (what == kScanLargest) most *= kProbeEvery;
                counters[kCntLargestBin] = most;
                if (largest) *largest = most;
            }
        }
    }
    cluster.sync();   // no CTA leaves while another reads its totals
}

// Four consecutive Gaussians per thread, 16-byte loads.  kFew: most of them take
// no part (depth slices), so ranks are read first and boxes one by one.  Bound
// by its scattered accesses, about one clock per lane and SM each: a bin start
// gathered and a record written per Gaussian that takes part.
template <bool kFew>
__global__ void __launch_bounds__(256)
k_bin_scatter(const uint32_t* __restrict__ keys, const uint32_t* __restrict__ ranks,
              const uint32_t* __restrict__ boxes, const uint32_t* __restrict__ bins,
              const uint32_t* __restrict__ bin_limit, const FrameParams* __restrict__ fp, BinMap map,
              int64_t n, uint4* __restrict__ out, uint32_t* __restrict__ status) {
    pdl_prologue();
    const uint32_t base = bin_base(fp->cam.near_z), limit = bin_limit ? *bin_limit : 0xFFFFFFFFu;
    const int64_t i0 = 4 * ((int64_t)blockIdx.x * 256 + threadIdx.x);
    if (i0 >= n) return;
    uint32_t k[4] = {0u, 0u, 0u, 0u}, r[4], x[4];
    if (i0 + 4 <= n) {
        const uint4 b = *reinterpret_cast<const uint4*>(ranks + i0);
        r[0] = b.x; r[1] = b.y; r[2] = b.z; r[3] = b.w;
        if (kFew && (r[0] & r[1] & r[2] & r[3]) == kNoRank) return;   // no rank is that large
        const uint4 a = *reinterpret_cast<const uint4*>(keys + i0);
        k[0] = a.x; k[1] = a.y; k[2] = a.z; k[3] = a.w;
        if (!kFew) {
            const uint4 c = *reinterpret_cast<const uint4*>(boxes + i0);
            x[0] = c.x; x[1] = c.y; x[2] = c.z; x[3] = c.w;
        }
    } else {
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            r[q] = i0 + q < n ? ranks[i0 + q] : kNoRank;
            if (i0 + q < n) k[q] = keys[i0 + q];
            if (!kFew && i0 + q < n) x[q] = boxes[i0 + q];
        }
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        if (r[q] == kNoRank) continue;
        const uint32_t bin = bin_of(k[q], base, map);
        if (bin >= limit) continue;
        const uint32_t pos = bins[bin] + r[q];
        if ((int64_t)pos < n) out[pos] = make_uint4(k[q], (uint32_t)(i0 + q), kFew ? boxes[i0 + q] : x[q], 0u);
        else atomicOr(status, kErrRange);
    }
}

// ---------------------------------------------------------------------------
// Window sort and run scan.
// ---------------------------------------------------------------------------
struct alignas(16) WindowShared {
    union {
        uint2 rec[kWinCap];                      // (key, index) grouped by sub-bin
        struct {
            uint32_t idx[kWinCap];               // the window in depth order
            uint32_t box[kWinCap];
        } out;
        uint32_t warp_cnt[kWinWarps][kRadix];    // large windows: radix ranking
    } u;
    union {
        uint32_t pair[kSub / 2 + 4];             // sub-bin counts, then starts, two 16-bit words each
        uint32_t off[kWinCap];                   // run offsets from the window's first run
        uint32_t run[kRadix];                    // large windows: next position of each digit
    } c;
    uint32_t w0[kWinWarps], w1[kWinWarps];
    unsigned long long sum;                      // large windows: column runs
    uint32_t ticket, prefix, total;              // total: the window's column runs
};
static_assert(kWinCap * 2 == kSub && kWinCap < (1 << 16), "16-bit starts, thread t scans 16 sub-bins");

__device__ __forceinline__ uint32_t box_runs(uint32_t box) { return ((box >> 16) & 0xFFu) + 1u; }

// Exclusive scan over the block of one value per thread; `total` the sum.
__device__ __forceinline__ uint32_t win_scan(uint32_t v, uint32_t* s_w, uint32_t& total) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) s_w[warp] = x;
    __syncthreads();
    uint32_t base = 0;
    total = 0;
#pragma unroll
    for (int w = 0; w < kWinWarps; ++w) {
        const uint32_t s = s_w[w];
        base += w < warp ? s : 0u;
        total += s;
    }
    __syncthreads();
    return base + x - v;
}

// Window [lo, lo + m), m <= kWinCap, into sm.u.out in depth order.  Its key
// range is cut into at most kSub sub-bins, filled with shared-memory atomics; a
// Gaussian's place is its sub-bin's start plus the members before it (a window
// has about kSub / 4 Gaussians, so most are alone in their sub-bin).  False, and
// nothing done, if a sub-bin has more than kCrowded members (many equal depths).
__device__ __forceinline__ bool sort_on_chip(WindowShared& sm, const uint4* __restrict__ recs, uint32_t lo,
                                             int m) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    uint4 rec[kWinItems];   // key, index, box, then the place
    uint32_t kmin = 0xFFFFFFFFu, kmax = 0u;
#pragma unroll
    for (int q = 0; q < kWinItems; ++q) {
        const int s = q * kWinThreads + tid;
        if (s < m) rec[q] = recs[lo + s];
    }
    uint4* c4 = reinterpret_cast<uint4*>(sm.c.pair) + 2 * tid;
    c4[0] = make_uint4(0u, 0u, 0u, 0u);
    c4[1] = make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
    for (int q = 0; q < kWinItems; ++q) {
        if (q * kWinThreads + tid < m) {
            kmin = min(kmin, rec[q].x);
            kmax = max(kmax, rec[q].x);
        }
    }
    kmin = __reduce_min_sync(0xffffffffu, kmin);
    kmax = __reduce_max_sync(0xffffffffu, kmax);
    if (lane == 0) {
        sm.w0[warp] = kmin;
        sm.w1[warp] = kmax;
    }
    __syncthreads();
#pragma unroll
    for (int w = 0; w < kWinWarps; ++w) {
        kmin = min(kmin, sm.w0[w]);
        kmax = max(kmax, sm.w1[w]);
    }
    const int bits = 32 - __clz(kmax - kmin);
    const int shift = bits > kSubBits ? bits - kSubBits : 0;
#pragma unroll
    for (int q = 0; q < kWinItems; ++q) {
        if (q * kWinThreads + tid < m) {   // .w: arrival rank in the sub-bin
            const uint32_t sub = (rec[q].x - kmin) >> shift, half = 16u * (sub & 1u);
            rec[q].w = (atomicAdd(&sm.c.pair[sub >> 1], 1u << half) >> half) & 0xFFFFu;
        }
    }
    __syncthreads();
    bool crowded;
    {
        uint4 a = c4[0], b = c4[1];
        uint32_t* v[8] = {&a.x, &a.y, &a.z, &a.w, &b.x, &b.y, &b.z, &b.w};
        uint32_t sum = 0, most = 0;
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            sum += (*v[j] & 0xFFFFu) + (*v[j] >> 16);
            most = max(most, max(*v[j] & 0xFFFFu, *v[j] >> 16));
        }
        crowded = most > kCrowded;
        uint32_t total;
        uint32_t run = win_scan(sum, sm.w0, total);
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const uint32_t lo16 = *v[j] & 0xFFFFu, hi16 = *v[j] >> 16;
            *v[j] = run | ((run + lo16) << 16);
            run += lo16 + hi16;
        }
        c4[0] = a;
        c4[1] = b;
        if (tid == 0) sm.c.pair[kSub / 2] = (uint32_t)m;
    }
    if (__syncthreads_or(crowded)) return false;
    const uint16_t* start = reinterpret_cast<const uint16_t*>(sm.c.pair);
#pragma unroll
    for (int q = 0; q < kWinItems; ++q) {
        if (q * kWinThreads + tid < m) {   // .w: slot
            rec[q].w += start[(rec[q].x - kmin) >> shift];
            sm.u.rec[rec[q].w] = make_uint2(rec[q].x, rec[q].y);
        }
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < kWinItems; ++q) {
        if (q * kWinThreads + tid < m) {   // .w: place in the window
            const uint32_t sub = (rec[q].x - kmin) >> shift;
            const uint32_t s0 = start[sub], s1 = start[sub + 1];
            if (s1 - s0 > 1u) {
                uint32_t place = s0;
                for (uint32_t j = s0; j < s1; ++j) {
                    const uint2 r = sm.u.rec[j];
                    place += (r.x < rec[q].x || (r.x == rec[q].x && r.y < rec[q].y)) ? 1u : 0u;
                }
                rec[q].w = place;
            }
        }
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < kWinItems; ++q) {
        if (q * kWinThreads + tid < m) {
            sm.u.out.idx[rec[q].w] = rec[q].y;
            sm.u.out.box[rec[q].w] = rec[q].z;
        }
    }
    __syncthreads();
    return true;
}

// A window of more than kWinCap Gaussians (one bin that large: very many
// Gaussians at nearly one depth) or a crowded one: a least-significant-digit radix sort by
// (key, index) of the CTA alone, skipping the digits that all its Gaussians
// share.  The window's 16-byte records make room for two buffers of (key, index).
// Returns the one holding the result.
__device__ const uint2* sort_large(WindowShared& sm, uint4* recs, uint32_t m) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    uint2 *src = reinterpret_cast<uint2*>(recs), *dst = src + m;
    const uint4 first = recs[0];
    uint32_t dk = 0, di = 0;
    for (uint32_t c0 = 0; c0 < m; c0 += kWinThreads) {   // (key, index) into the first half, in place
        const uint32_t s = c0 + tid;
        const uint4 r = s < m ? recs[s] : first;
        dk |= r.x ^ first.x;
        di |= r.y ^ first.y;
        __syncthreads();   // what is overwritten has been read
        if (s < m) src[s] = make_uint2(r.x, r.y);
        __syncthreads();
    }
    dk = __reduce_or_sync(0xffffffffu, dk);
    di = __reduce_or_sync(0xffffffffu, di);
    if (lane == 0) {
        sm.w0[warp] = dk;
        sm.w1[warp] = di;
    }
    __syncthreads();
    for (int w = 0; w < kWinWarps; ++w) {
        dk |= sm.w0[w];
        di |= sm.w1[w];
    }
    uint32_t* run = sm.c.run;
    for (int pass = 0; pass < 8; ++pass) {
        const int shift = 8 * (pass & 3);
        if ((((pass < 4 ? di : dk) >> shift) & 0xFFu) == 0u) continue;
        auto digit = [&](uint2 r) { return ((pass < 4 ? r.y : r.x) >> shift) & 0xFFu; };
        __syncthreads();
        run[tid] = 0u;
        __syncthreads();
        for (uint32_t s = tid; s < m; s += kWinThreads) atomicAdd(&run[digit(src[s])], 1u);
        __syncthreads();
        uint32_t total;
        run[tid] = win_scan(run[tid], sm.w0, total);
        for (uint32_t c0 = 0; c0 < m; c0 += kWinThreads * kLargeItems) {
            for (int d = lane; d < kRadix; d += 32) sm.u.warp_cnt[warp][d] = 0u;
            __syncwarp();
            uint2 rec[kLargeItems];
            uint32_t at[kLargeItems];
#pragma unroll
            for (int q = 0; q < kLargeItems; ++q) {   // warp-striped, so the order is kept
                const uint32_t s = c0 + warp * (kLargeItems * 32) + q * 32 + lane;
                const bool in = s < m;
                rec[q] = in ? src[s] : make_uint2(0u, 0u);
                const uint32_t d = digit(rec[q]);
                uint32_t peers = __ballot_sync(0xffffffffu, in);
#pragma unroll
                for (int b = 0; b < kRadixBits; ++b) {
                    const uint32_t ones = __ballot_sync(0xffffffffu, (d >> b) & 1u);
                    peers &= ((d >> b) & 1u) ? ones : ~ones;
                }
                const uint32_t had = in ? sm.u.warp_cnt[warp][d] : 0u;
                at[q] = had + __popc(peers & ((1u << lane) - 1u));
                __syncwarp();
                if (in && lane == 31 - __clz(peers)) sm.u.warp_cnt[warp][d] = had + __popc(peers);
                __syncwarp();
            }
            __syncthreads();
            uint32_t p = run[tid];
            for (int w = 0; w < kWinWarps; ++w) {
                const uint32_t c = sm.u.warp_cnt[w][tid];
                sm.u.warp_cnt[w][tid] = p;
                p += c;
            }
            run[tid] = p;
            __syncthreads();
#pragma unroll
            for (int q = 0; q < kLargeItems; ++q) {
                const uint32_t s = c0 + warp * (kLargeItems * 32) + q * 32 + lane;
                if (s < m) dst[sm.u.warp_cnt[warp][digit(rec[q])] + at[q]] = rec[q];
            }
            __syncthreads();
        }
        uint2* other = src;
        src = dst;
        dst = other;
    }
    __syncthreads();
    return src;
}

// The parts of k_window_sort for a window that is not sorted on chip: its run total
// (of the unsorted records: the windows behind it wait for this, not for the sort),
// its order and boxes, and its run offsets.
__device__ __noinline__ void total_large(WindowShared& sm, const uint4* recs, uint32_t m) {
    if (threadIdx.x == 0) sm.sum = 0ull;
    __syncthreads();
    unsigned long long runs = 0;
#pragma unroll 4
    for (uint32_t s = threadIdx.x; s < m; s += kWinThreads) runs += box_runs(recs[s].z);
    atomicAdd(&sm.sum, runs);
    __syncthreads();
    if (threadIdx.x == 0) sm.total = (uint32_t)min(sm.sum, (unsigned long long)kSat);
}

__device__ __noinline__ void order_large(WindowShared& sm, uint4* recs, uint32_t m, const uint32_t* gbox,
                                         uint32_t* order, uint32_t* sorted_box) {
    const uint2* sorted = sort_large(sm, recs, m);
    for (uint32_t s = threadIdx.x; s < m; s += kWinThreads) {
        const uint32_t i = sorted[s].y;
        order[s] = i;
        sorted_box[s] = gbox[i];
    }
    __syncthreads();   // offsets_large reads the boxes
}

__device__ __noinline__ void offsets_large(WindowShared& sm, uint32_t lo, uint32_t m, const uint32_t* sorted_box,
                                           uint32_t prefix, int64_t capacity, uint32_t* offsets,
                                           uint32_t* chunk_first) {
    for (uint32_t p0 = 0; p0 < m; p0 += kWinThreads) {
        const uint32_t s = p0 + threadIdx.x;
        const uint32_t t = s < m ? box_runs(sorted_box[lo + s]) : 0u;
        uint32_t total;
        const uint32_t run = sat_add(prefix, win_scan(t, sm.w0, total));
        if (s < m) {
            offsets[lo + s] = run;
            mark_chunks(run, t, lo + s, capacity, chunk_first);
        }
        prefix = sat_add(prefix, total);
    }
}

__global__ void __launch_bounds__(kWinThreads, 4)
k_window_sort(uint4* recs, const uint32_t* __restrict__ win_lo, const uint32_t* __restrict__ gbox,
              int64_t n_max, int64_t capacity, uint32_t* order, uint32_t* sorted_box, uint32_t* offsets,
              uint32_t* __restrict__ chunk_first, unsigned long long* __restrict__ lookback, EpochRef eref,
              uint32_t* block, uint32_t* __restrict__ counters, uint32_t* __restrict__ slices,
              uint32_t* __restrict__ status, LookbackTest lt) {
    pdl_prologue();
    __shared__ WindowShared sm;
    const uint32_t epoch = (*eref.stage) * 8u + eref.pass;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t V = (uint32_t)min((int64_t)block[kCntVisible], n_max);
    const uint32_t windows = (V + (uint32_t)kWindow - 1u) / (uint32_t)kWindow;
    for (;;) {
        // Windows are taken in order, so a window's predecessors are done or running.
        if (tid == 0) sm.ticket = atomicAdd(block + kCntScanTicket, 1u);
        __syncthreads();
        const uint32_t w = sm.ticket;
        if (w >= windows) return;
        const uint32_t lo = min(win_lo[w], V), hi = min(max(win_lo[w + 1], lo), V), m = hi - lo;
        const bool on_chip = m <= (uint32_t)kWinCap && sort_on_chip(sm, recs, lo, (int)m);
        if (on_chip) {
            // Thread t's eight consecutive Gaussians: their run offsets from the
            // window's first run.
            uint32_t runs = 0, off[kWinItems];
            const uint4* b4 = reinterpret_cast<const uint4*>(sm.u.out.box) + 2 * tid;
            const uint4 a = b4[0], b = b4[1];
            const uint32_t box[kWinItems] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
#pragma unroll
            for (int q = 0; q < kWinItems; ++q) {
                off[q] = runs;
                if (kWinItems * tid + q < (int)m) runs += box_runs(box[q]);
            }
            uint32_t total;
            const uint32_t before = win_scan(runs, sm.w0, total);
            uint4* o4 = reinterpret_cast<uint4*>(sm.c.off) + 2 * tid;
            o4[0] = make_uint4(before + off[0], before + off[1], before + off[2], before + off[3]);
            o4[1] = make_uint4(before + off[4], before + off[5], before + off[6], before + off[7]);
            if (tid == 0) sm.total = total;
        } else {
            total_large(sm, recs + lo, m);
        }
        __syncthreads();
        if (warp == 0) {
            bool gave_up;
            const uint32_t excl = warp_lookback(lookback, w, sm.total, epoch, status, lt, &gave_up);
            if (lane == 0) {
                sm.prefix = excl;
                if (w + 1 == windows) block[kCntRuns] = sat_add(excl, sm.total);
                if (gave_up) {   // not a valid scan: the pair counts read as saturated, so every
                                 // later stage skips its work
                    counters[kCntPairs] = kSat;
                    if (slices) slices[kCntPairs] = slices[kCntSlots + kCntPairs] = kSat;
                }
            }
        } else if (on_chip) {   // meanwhile the other warps write the order out
            for (int s = tid - 32; s < (int)m; s += kWinThreads - 32) {
                order[lo + s] = sm.u.out.idx[s];
                sorted_box[lo + s] = sm.u.out.box[s];
            }
        }
        __syncthreads();
        if (on_chip) {
            for (int s = tid; s < (int)m; s += kWinThreads) {
                const uint32_t run = sat_add(sm.prefix, sm.c.off[s]);
                offsets[lo + s] = run;
                mark_chunks(run, box_runs(sm.u.out.box[s]), lo + s, capacity, chunk_first);
            }
        } else {
            order_large(sm, recs + lo, m, gbox, order + lo, sorted_box + lo);
            offsets_large(sm, lo, m, sorted_box, sm.prefix, capacity, offsets, chunk_first);
        }
        __syncthreads();   // the window is no longer read
    }
}

}  // namespace

BinMap bin_map(int64_t n) {
    BinMap m;
    m.shift = n <= (1 << 15) ? 14 : n <= (1 << 18) ? 13 : n <= (1 << 19) ? 12 : n <= (1 << 20) ? 11 : 10;
    m.count = (uint32_t)kBinOctaves << (23 - m.shift);
    return m;
}

int window_blocks_per_sm() {
    int b = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, k_window_sort, kWinThreads, 0) != cudaSuccess)
        return 1;
    return b > 0 ? b : 1;
}

void launch_bin_scan(uint32_t* bins, const BinMap& map, uint32_t* win_lo, BinScan what, uint32_t* counters,
                     uint32_t* slice_counters, const unsigned long long* sums, int64_t capacity,
                     uint32_t* largest, uint32_t* status, cudaStream_t stream) {
    // 1, 2 or 4 quads of bins a lane in 256 to 1024 threads, for 2^13 to 2^17 bins
    const uint32_t per_cta = map.count / kScanCluster;
    const int quads = per_cta <= 1024 ? 1 : per_cta <= 2048 ? 2 : 4;
    auto* kernel = quads == 1 ? k_bin_scan<1> : quads == 2 ? k_bin_scan<2> : k_bin_scan<4>;
    launch_pdl(kernel, kScanCluster, per_cta / (4 * quads), 0, stream, bins, win_lo, (int)what, counters,
               slice_counters, sums, capacity, largest, status);
}

void launch_bin_scatter(const uint32_t* keys, const uint32_t* ranks, const uint32_t* boxes,
                        const uint32_t* bins, const uint32_t* bin_limit, bool few, const FrameParams* fp,
                        const BinMap& map, int64_t n, uint4* out, uint32_t* status, cudaStream_t stream) {
    if (n <= 0) return;
    launch_pdl(few ? k_bin_scatter<true> : k_bin_scatter<false>, (unsigned)((n + 1023) / 1024), 256, 0, stream,
               keys, ranks, boxes, bins, bin_limit, fp, map, n, out, status);
}

void launch_window_sort(uint4* recs, const uint32_t* win_lo, const uint32_t* gbox, int64_t n,
                        int64_t capacity, uint32_t* order, uint32_t* sorted_box, uint32_t* offsets,
                        uint32_t* chunk_first, unsigned long long* lookback, EpochRef epoch,
                        uint32_t* block, uint32_t* counters, uint32_t* slice_counters, uint32_t* status,
                        int grid, cudaStream_t stream) {
    if (n <= 0) return;
    const int64_t most = (n + kWindow - 1) / kWindow;
    launch_pdl(k_window_sort, (unsigned)(most < grid ? most : grid), kWinThreads, 0, stream, recs, win_lo, gbox,
               n, capacity, order, sorted_box, offsets, chunk_first, lookback, epoch, block, counters,
               slice_counters, status, lookback_test());
}

}  // namespace adr
