"""The image loss's means at the ends of the range and in all their bits, which are
those of FP64 sums over the pixels."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _stats(img, ref, want_grad=False):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2409_08669_gb300.raster import image_loss
    stats, grad = image_loss(torch.from_numpy(img).cuda(), torch.from_numpy(ref).cuda(), 0.44, 0.11, want_grad=want_grad)
    return stats.cpu().numpy(), grad


@pytest.mark.parametrize("value", [float("inf"), -float("inf")])
@pytest.mark.parametrize("c,h,w,at", [(1, 1, 1, (0, 0, 0)), (3, 60, 70, (1, 58, 3)), (1, 54, 32, (0, 53, 31))])
def test_an_infinite_pixel_gives_an_infinite_mean(value, c, h, w, at):
    rng = np.random.default_rng(h)
    img, ref = rng.random((c, h, w), dtype=np.float32), rng.random((c, h, w), dtype=np.float32)
    img[at] = value
    assert _stats(img, ref)[0][0] == math.inf


@pytest.mark.parametrize("value", [3e38, 1e36])
def test_a_sum_beyond_32_bits_is_finite(value):
    img, ref = np.full((2, 60, 70), value, np.float32), np.zeros((2, 60, 70), np.float32)
    assert abs(_stats(img, ref)[0][0] / float(np.float32(value)) - 1.0) <= 1e-12


@pytest.mark.parametrize("c,h,w", [(1, 54, 32), (1, 7, 29), (3, 300, 500)])
def test_the_mean_difference_has_64_bits(c, h, w):
    """Of differences over 40 octaves.  Each value passes at most 7 + 5 + 8 additions and its tile's one to memory, each
    rounded to 2^-53 of a partial sum that is at most the whole."""
    rng = np.random.default_rng(w)
    img = np.exp2(rng.uniform(-30, 10, (c, h, w))).astype(np.float32)
    ref = np.zeros_like(img)
    exact = math.fsum(img.reshape(-1).astype(np.float64)) / img.size
    tiles = c * -(-h // 54) * -(-w // 32)
    assert abs(_stats(img, ref)[0][0] - exact) <= (20 + tiles + 1) * 2.0 ** -53 * exact


@pytest.mark.parametrize("hw,top", [(136 * 120, 60), (300 * 200 + 1, 300), (1280 * 720, 2000)])
def test_the_load_gradient_is_the_rounded_64_bit_one(hw, top):
    """Its float pairs keep 48 bits before the one rounding to FP32: of the loads of frames (whole numbers to a few
    thousand) no value lies near enough to a rounding's middle to fall on the other side."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2409_08669_gb300.raster import Rasterizer
    load = np.minimum(np.random.default_rng(hw).gamma(2.0, top / 6, hw), top).astype(np.int32)
    rast = Rasterizer(max_gaussians=16, pair_capacity=16, max_width=16, max_height=16)
    try:
        stats, grad = rast.load_loss(torch.from_numpy(load).cuda(), weight=1.0)
        mean, std = stats.cpu().numpy()
        grad = grad.cpu().numpy()
    finally:
        rast.close()
    assert np.array_equal(grad, ((load.astype(np.float64) - mean) * (1.0 / (hw * std))).astype(np.float32))
