"""The choice of a frame's depth order (csrc/depth_sort.h: host code, compiled here
with g++), from the largest depth bin of earlier frames."""
import os
import subprocess

import pytest

_SRC = r"""
#include <cstdio>
#include <cstdlib>
#include "depth_sort.h"
using namespace adr;
// argv: the Gaussians, then pairs of (scene, largest bin its frame has): frames that share one buffer's word, as
// the requests on a serving slot do.  Prints each frame's choice.
int main(int argc, char** argv) {
    DepthSortChoice scene[4];
    uint32_t word = 0xABCDu;   // not written yet
    const long long n = std::atoll(argv[1]);
    for (int k = 2; k + 1 < argc; k += 2) {
        DepthSortChoice& s = scene[std::atoi(argv[k])];
        const DepthSort used = s.next(n);
        if (used != kSortRadix) word = (uint32_t)std::atoll(argv[k + 1]);
        s.completed(used, word);
        std::printf("%d ", (int)used);
    }
    return 0;
}
"""
BINS, RADIX, PROBE = 0, 1, 2


@pytest.fixture(scope="module")
def choices(tmp_path_factory):
    d = tmp_path_factory.mktemp("depth_sort")
    (d / "choice.cpp").write_text(_SRC)
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    subprocess.run(["g++", "-std=c++17", f"-I{os.path.join(root, 'paper_2409_08669_gb300', 'csrc')}",
                    str(d / "choice.cpp"), "-o", str(d / "choice")], check=True)

    def run(frames, n=3_000_000):
        args = [str(n)] + [str(v) for f in frames for v in f]
        return [int(v) for v in subprocess.run([str(d / "choice"), *args], capture_output=True, text=True,
                                               check=True).stdout.split()]
    return run


def test_a_flat_scene_keeps_the_radix_sort_beside_an_ordinary_one(choices):
    """Two scenes on one slot: a radix frame leaves the other scene's word, which says nothing about its own bins."""
    frames = [(0, 100_000), (1, 50)] * 200
    got = choices(frames)
    flat, ordinary = got[0::2], got[1::2]
    assert ordinary[1:] == [BINS] * 199
    assert BINS not in flat[1:]
    assert [k for k, c in enumerate(flat[1:], 1) if c == PROBE] == [64, 128, 192]


@pytest.mark.parametrize("largest,sort", [(50, BINS), (1000, BINS), (1500, BINS), (2300, RADIX), (5000, RADIX), (1_000_000, RADIX)])
def test_the_faster_sort_by_the_largest_bin(choices, largest, sort):
    """The line lies where the two sorts were measured to cross (1500 to 2200 Gaussians in a bin)."""
    got = choices([(0, largest)] * 10)
    assert got[2:] == [sort] * 8


def test_a_first_frame_is_measured_beside_the_radix_sort(choices):
    """Nothing is known of a scene before its first frame: the radix sort's time does not depend on its depths."""
    assert choices([(0, 50), (1, 100_000)] * 3) == [PROBE, PROBE, BINS, RADIX, BINS, RADIX]
    assert choices([(0, 50)] * 3, n=1536) == [BINS, BINS, BINS]      # no bin can hold more
