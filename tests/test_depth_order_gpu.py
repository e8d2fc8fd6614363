"""The depth order of the Gaussians (bins.cu; the radix sort of sort.cu where
very many share a bin), at the sizes where its windows, bins and dispatch can go
wrong.  All Gaussians of a frame cover the one tile of a 16x16 image, so the
tile's list is the whole order: the FP32 depth bits ascending, equal depths by
Gaussian index."""
import numpy as np
import pytest

from paper_2409_08669_gb300 import scenes as S

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _depths(kind, n, rng):
    if kind == "spread":            # ordinary depths over a few octaves
        return rng.uniform(0.5, 8.0, n)
    if kind == "equal":             # one depth: ordered by index alone
        return np.full(n, 3.0)
    if kind == "ties":              # 50 distinct depths
        return 2.0 + rng.integers(0, 50, n) / 64.0
    if kind == "wall":              # one bin, distinct depths
        return 4.0 + rng.uniform(0.0, 1e-4, n)
    if kind == "mixed":             # a wall of half the Gaussians among ordinary depths
        return np.where(rng.random(n) < 0.5, 4.0 + rng.uniform(0.0, 1e-4, n), rng.uniform(0.5, 8.0, n))
    assert kind == "octaves"        # nearer than the first bin to beyond the last
    return np.exp(rng.uniform(np.log(2e-3), np.log(4e4), n))


@pytest.mark.parametrize("kind,n", [
    ("spread", 1), ("spread", 2047), ("spread", 2048), ("spread", 2049), ("spread", 32768), ("spread", 32769),
    ("spread", 300_001), ("equal", 4096), ("equal", 4097), ("equal", 20_000), ("ties", 30_000), ("wall", 4097),
    ("wall", 40_000), ("mixed", 9_000), ("octaves", 50_000)])
def test_list_is_by_depth_then_index(kind, n):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2409_08669_gb300.raster import Rasterizer, upload
    rng = np.random.default_rng(n)
    depth = _depths(kind, n, rng)
    scene = S.tiny_scene(1, n=n)
    scene.means[:] = np.stack([np.zeros(n), np.zeros(n), depth], axis=1).astype(np.float32)
    scene.scales[:] = (0.05 * depth[:, None]).astype(np.float32)     # a few pixels at any depth
    scene.opac[:] = 0.5
    cam = S.look_at((0, 0, 0), target=(0, 0, 1), width=16, height=16, near=1e-3)
    key = (scene.means[:, 2] + np.float32(0)).view(np.uint32).astype(np.uint64)   # the view is the identity
    want = np.lexsort((np.arange(n), key))
    rast = Rasterizer(max_gaussians=n, pair_capacity=max(n, 16), max_width=16, max_height=16)
    try:
        params = upload(scene)
        images = []
        for _ in range(3):          # the later frames take the sort that the first one's bins call for
            img, _, load = rast.forward(params, cam, S.Settings(t_min=0.0))
            keys, vals = rast.read_pairs()
            assert rast.sync_status() == 0
            assert np.array_equal(vals.astype(np.int64), want)
            assert np.array_equal(keys, key[want])
            images.append((img.clone(), load.clone()))
        for img, load in images[1:]:
            assert torch.equal(img, images[0][0]) and torch.equal(load, images[0][1])
    finally:
        rast.close()
