// Which depth order a frame is built with, from what earlier frames measured.
// Host code without CUDA calls, so the choice is testable without a GPU.
#pragma once

#include <stdint.h>

namespace adr {

// How a frame orders its Gaussians by depth: by bins (bins.cu), or by the
// radix sort (sort.cu), with or without a depth histogram beside it.  Both give
// the same order; the radix sort is the faster one where many Gaussians lie at
// nearly one depth: a window of more than 2048 is sorted by one CTA, and a bin is
// counted by atomics on one address.  Frames at 1280x720 of Gaussians about one plane, bins /
// radix sort, by the largest bin: 10k, 1331: 80 / 116 us; 30k, 1345: 83 / 133; 300k, 1049:
// 267 / 289; 1M, 1765: 383 / 358; 100k, 2252: 214 / 208; 300k, 3422: 353 / 291; 10k,
// 4287: 133 / 116; 1M, 5655: 737 / 361.  Scenes that spread over octaves have at
// most 1000 (3M Gaussians).
enum DepthSort : int { kSortBins = 0, kSortRadix = 1, kSortRadixProbe = 2 };
constexpr uint32_t kRadixBin = 1536;
constexpr uint32_t kRadixProbe = 64;   // a histogram every 64th radix frame

// One per context, served scene or allocation-free device.
struct DepthSortChoice {
    uint32_t largest_bin = 0;          // of the last completed frame that had a histogram
    uint32_t probe_in = kRadixProbe;   // radix frames until the next one with a histogram

    DepthSort next() {
        if (largest_bin <= kRadixBin) {
            probe_in = kRadixProbe;
            return kSortBins;
        }
        if (--probe_in > 0) return kSortRadix;
        probe_in = kRadixProbe;
        return kSortRadixProbe;
    }
    // A frame built with `used` completed and left `largest` in its buffers' word: a radix
    // frame without a histogram wrote none, so the word may be another scene's.
    void completed(DepthSort used, uint32_t largest) {
        if (used != kSortRadix) largest_bin = largest;
    }
};

}  // namespace adr
