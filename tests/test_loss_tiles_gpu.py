"""The image loss and the load loss at the sizes where their tiles and vector
loads can go wrong: one pixel, edges of the 32x54 tile, planes that are not a
multiple of 16 bytes; loads of any sign and size."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("c,h,w", [(1, 1, 1), (1, 53, 31), (3, 54, 32), (2, 55, 33), (1, 108, 65), (3, 7, 301)])
def test_image_loss_at_tile_edges(c, h, w):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from oracle import ssim as ossim
    from paper_2409_08669_gb300.raster import image_loss
    rng = np.random.default_rng(100 * h + w)
    img = rng.random((c, h, w), dtype=np.float32)
    ref = np.clip(img + rng.normal(0.0, 0.1, img.shape), 0, 1).astype(np.float32)
    l1, ms, g = ossim.image_loss(img, ref, 0.44, 0.11)
    stats, grad = image_loss(torch.from_numpy(img).cuda(), torch.from_numpy(ref).cuda(), 0.44, 0.11)
    stats, grad = stats.cpu().numpy(), grad.cpu().numpy()
    # FP32 moments (~1e-7 absolute) over C2 = 9e-4: ~1e-4 relative on S where the
    # variance is small; 2e-5 on its mean and 2e-3 of the largest gradient bound that
    assert abs(stats[0] - l1) <= 1e-6 * max(l1, 1.0) and abs(stats[1] - ms) <= 2e-5
    assert np.abs(grad - g).max() <= 2e-3 * np.abs(g).max()


@pytest.mark.parametrize("hw,offset,top", [(1, 0, 50), (3, 0, 50), (1023, 1, 300), (4096, 0, 1), (921_601, 3, 2000),
                                            (2048, 2, 2**31 - 1)])
def test_load_loss_moments_and_gradient(hw, offset, top):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2409_08669_gb300.raster import Rasterizer
    rng = np.random.default_rng(hw)
    host = rng.integers(-top if top > 10_000 else 0, top, size=hw + offset, endpoint=True).astype(np.int32)
    load = torch.from_numpy(host).cuda()[offset:]          # not 16-byte aligned for every offset
    v = host[offset:].astype(np.float64)
    rast = Rasterizer(max_gaussians=16, pair_capacity=16, max_width=16, max_height=16)
    try:
        stats, grad = rast.load_loss(load, weight=0.45)
        stats, grad = stats.cpu().numpy(), grad.cpu().numpy()
    finally:
        rast.close()
    mean = v.mean()
    std = v.std()
    # exact sums; the variance as a difference of FP64 terms keeps 1e-16 of E[l^2]
    assert abs(stats[0] - mean) <= 1e-12 * max(1.0, abs(mean))
    assert abs(stats[1] ** 2 - std ** 2) <= 1e-12 * max(1.0, (v ** 2).mean())
    if std > 0:
        want = 0.45 * (v - mean) / (hw * std)
        # rounded once to FP32, with float pairs before it
        assert np.abs(grad - want).max() <= 2e-7 * np.abs(want).max() + 1e-12
