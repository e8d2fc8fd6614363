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
// That histogram counts every 8th Gaussian: of all, atomics on one address took 435 us
// of a 1016 us frame (3M Gaussians within 1% of one depth).
constexpr uint32_t kProbeEvery = 8;
constexpr uint32_t kUnknownBin = 0xFFFFFFFFu;

// One per context, served scene or allocation-free device.
struct DepthSortChoice {
    uint32_t largest_bin = kUnknownBin;   // of the last completed frame that had a histogram
    uint32_t probe_in = kRadixProbe;   // radix frames until the next one with a histogram

    // The sort of a frame of n Gaussians.  Until a frame has been measured the radix sort, whose
    // time does not depend on the depths: a first frame of 3M Gaussians, over octaves to one
    // depth, took 0.43 to 33 ms by bins, 0.58 to 0.82 by the passes.
    DepthSort next(int64_t n) {
        if (largest_bin <= kRadixBin || n <= (int64_t)kRadixBin) {
            probe_in = kRadixProbe;
            return kSortBins;
        }
        if (largest_bin == kUnknownBin) return kSortRadixProbe;
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
