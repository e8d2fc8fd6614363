"""The depth order of scenes at nearly one depth, after frames of ordinary ones (the
choice of the sort goes by earlier frames, so this frame's bins hold them all)."""
import numpy as np
import pytest

from paper_2409_08669_gb300 import scenes as S

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _scene(depth, seed=1):
    n = len(depth)
    scene = S.tiny_scene(seed, n=n)
    scene.means[:] = np.stack([np.zeros(n), np.zeros(n), depth], axis=1).astype(np.float32)
    scene.scales[:] = (0.05 * np.asarray(depth)[:, None]).astype(np.float32)     # a few pixels at any depth
    scene.opac[:] = 0.5
    return scene


def _frames(n):
    """An ordinary scene's parameters and depths of n Gaussians, and the camera that sees their order in one tile."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    cam = S.look_at((0, 0, 0), target=(0, 0, 1), width=16, height=16, near=1e-3)
    return _scene(np.random.default_rng(n).uniform(0.5, 8.0, n)), cam


@pytest.fixture
def expiry():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2409_08669_gb300 import _lib
    yield _lib.adr_test_lookback_expiry
    _lib.adr_test_lookback_expiry(-1)


def test_windows_do_not_wait_for_the_sort_of_a_large_one(expiry):
    """300k Gaussians in one bin: its sort takes a few ms, its run total a few percent of that, and the windows behind it
    wait for the total only (1500 polls are under 1.5 ms; no chunk is withheld)."""
    from paper_2409_08669_gb300.raster import Rasterizer, upload
    n = 300_000
    ordinary, cam = _frames(n)
    flat = _scene(np.full(n, 3.0))
    st = S.Settings(t_min=0.0)
    rast = Rasterizer(max_gaussians=n, pair_capacity=n, max_width=16, max_height=16)
    try:
        for _ in range(2):
            rast.forward(upload(ordinary), cam, st)
            assert rast.sync_status() == 0
        expiry(1 << 20, 1500)
        rast.forward(upload(flat), cam, st)
        assert rast.sync_status() == 0
        assert np.array_equal(rast.read_pairs()[1], np.arange(n))
    finally:
        rast.close()


def _order_is_right(rast, params, depth, cam, st):
    rast.forward(params, cam, st)
    vals = rast.read_pairs()[1].astype(np.int64)
    assert rast.sync_status() == 0
    return np.array_equal(vals, np.lexsort((np.arange(len(depth)), depth.astype(np.float32).view(np.uint32))))


@pytest.mark.parametrize("n,equal", [(2000, 2000), (1025, 130), (1500, 127), (2040, 1000)])
def test_equal_depths_in_a_window(n, equal):
    """Windows that fit on chip, `equal` of whose Gaussians have one depth (the others a few octaves about it): ordered by
    index, and in no more than three times an ordinary frame's time (comparing each with all took 3.5 times at 2000)."""
    from paper_2409_08669_gb300.raster import Rasterizer, upload
    ordinary, cam = _frames(n)
    depth = np.random.default_rng(equal).uniform(0.5, 8.0, n)
    depth[np.random.default_rng(n).permutation(n)[:equal]] = 3.0
    st = S.Settings(t_min=0.0)
    rast = Rasterizer(max_gaussians=n, pair_capacity=1 << 16, max_width=16, max_height=16)
    try:
        same, spread = upload(_scene(depth)), upload(ordinary)
        us = {}
        for name, params in (("spread", spread), ("same", same)):
            for _ in range(5):
                rast.forward(params, cam, st)
            best = []
            for _ in range(5):
                e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
                e[0].record()
                for _ in range(10):
                    rast.forward(params, cam, st)
                e[1].record()
                torch.cuda.synchronize()
                best.append(e[0].elapsed_time(e[1]) * 100)
            us[name] = min(best)
        assert _order_is_right(rast, same, depth, cam, st)
        assert us["same"] <= 3 * us["spread"], us
    finally:
        rast.close()


@pytest.mark.parametrize("n", [20_001, 20_002, 20_003, 20_004])
def test_radix_frames_of_odd_sizes(n):
    """The radix passes' buffers in a workspace of any number of Gaussians (they are read 16 bytes at a time)."""
    from paper_2409_08669_gb300.raster import Rasterizer, upload
    _, cam = _frames(n)
    depth = np.full(n, 3.0)
    depth[::5] = np.random.default_rng(n).uniform(0.5, 8.0, len(depth[::5]))
    rast = Rasterizer(max_gaussians=n, pair_capacity=n, max_width=16, max_height=16)
    try:
        params = upload(_scene(depth))
        for _ in range(3):
            assert _order_is_right(rast, params, depth, cam, S.Settings(t_min=0.0))
    finally:
        rast.close()


@pytest.mark.parametrize("n,kind", [(4097, "equal"), (20_001, "equal"), (9_000, "mixed"), (40_001, "wall"), (30_000, "ties")])
def test_large_windows_after_an_ordinary_frame(n, kind):
    """A frame that was expected to have no large bin sorts it in its window."""
    from paper_2409_08669_gb300.raster import Rasterizer, upload
    ordinary, cam = _frames(n)
    rng = np.random.default_rng(n + 1)
    wall = 4.0 + rng.uniform(0.0, 1e-4, n)
    depth = {"equal": np.full(n, 3.0), "wall": wall, "mixed": np.where(rng.random(n) < 0.5, wall, rng.uniform(0.5, 8.0, n)),
             "ties": 2.0 + rng.integers(0, 5, n) / 64.0}[kind]
    st = S.Settings(t_min=0.0)
    rast = Rasterizer(max_gaussians=n, pair_capacity=n, max_width=16, max_height=16)
    try:
        for _ in range(2):
            rast.forward(upload(ordinary), cam, st)
            assert rast.sync_status() == 0
        for _ in range(2):
            assert _order_is_right(rast, upload(_scene(depth)), depth, cam, st)
    finally:
        rast.close()
