"""The training path's float loads and loss value, which the kernels write
themselves, against the separate passes they stand for: Render's float loads and
its integer ones, the load loss of either, and the image loss as a sum of its terms."""
import numpy as np
import pytest

from paper_2409_08669_gb300 import scenes as S

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _rast(n=2000, w=130, h=75):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2409_08669_gb300.raster import Rasterizer
    return Rasterizer(max_gaussians=n, pair_capacity=1 << 20, max_width=w, max_height=h)


@pytest.mark.parametrize("slices,split", [(0, 0), (1, 0), (1, 1)])
def test_render_writes_the_loads_as_floats(slices, split):
    from paper_2409_08669_gb300.raster import upload
    rast = _rast()
    try:
        rast.set_depth_slices(slices)
        rast.set_tile_split(split)
        params = upload(S.tiny_scene(3, n=2000))
        cam, st = S.look_at((0, 0.2, -2.5), width=130, height=75), S.Settings()
        img, t_final, load = rast.forward(params, cam, st)
        img_f, t_f, load_f = rast.forward(params, cam, st, load_dtype=torch.float32)
        assert load_f.dtype == torch.float32 and torch.equal(load_f, load.to(torch.float32))
        assert torch.equal(img, img_f) and torch.equal(t_final, t_f)
        with pytest.raises(ValueError):
            rast.render(load_dtype=torch.int64)
    finally:
        rast.close()


def test_a_frame_after_a_backward_is_not_sliced():
    from paper_2409_08669_gb300.raster import upload
    rast = _rast()
    try:
        params = upload(S.tiny_scene(3, n=2000))
        cam, st = S.look_at((0, 0.2, -2.5), width=130, height=75), S.Settings()
        frames, sliced = [], []
        for backward in (True, True, False, False):
            img, t_final, load = rast.forward(params, cam, st)
            frames.append((img, t_final, load))
            sliced.append(rast.frame_counts()["sliced"])
            if backward:
                rast.backward(params, torch.ones_like(img))
        assert sliced[:3] == [1, 0, 0]      # the first frame measures, two follow a backward
        rast.set_depth_slices(rast.SLICES_ALWAYS)
        rast.backward(params, torch.ones_like(img))
        frames.append(rast.forward(params, cam, st))
        assert rast.frame_counts()["sliced"] == 1
        for frame in frames[1:]:
            assert all(torch.equal(a, b) for a, b in zip(frame, frames[0]))
    finally:
        rast.close()


@pytest.mark.parametrize("hw,offset", [(1, 0), (3, 0), (1023, 1), (4096, 2), (921_601, 3)])
def test_load_loss_of_floats_is_that_of_the_rounded_loads(hw, offset):
    rast = _rast()
    try:
        rng = np.random.default_rng(hw)
        whole = rng.integers(0, 2000, hw + offset)
        off = rng.choice([0.0, 0.25, -0.25, 0.5], hw + offset)       # halves go to the even neighbour
        load = torch.from_numpy((whole + off).astype(np.float32)).cuda()[offset:]
        std, grad = rast.load_loss_float(load, 0.45)
        stats, want = rast.load_loss(load.round().to(torch.int32), 0.45)
        assert torch.equal(std, stats[1].to(torch.float32)) and torch.equal(grad, want)
    finally:
        rast.close()


@pytest.mark.parametrize("c,h,w,w_l1,w_ssim", [(1, 1, 1, 0.8, 0.2), (3, 55, 33, 0.44, 0.11), (2, 108, 65, 0.0, 1.0)])
def test_image_loss_value_is_the_sum_of_its_terms(c, h, w, w_l1, w_ssim):
    _rast().close()
    from paper_2409_08669_gb300.autograd import l1_ssim_loss
    from paper_2409_08669_gb300.raster import image_loss
    g = torch.Generator("cuda").manual_seed(h)
    ref = torch.rand(c, h, w, generator=g, device="cuda")
    img = (ref + 0.1 * torch.randn(c, h, w, generator=g, device="cuda")).requires_grad_(True)
    value = torch.empty((), device="cuda")
    stats, grad = image_loss(img.detach(), ref, w_l1, w_ssim, value=value)
    assert torch.equal(value, (w_l1 * stats[0] + w_ssim * (1.0 - stats[1])).to(torch.float32))
    loss = l1_ssim_loss(img, ref, w_l1, w_ssim)
    (2.0 * loss).backward()
    # the sums' atomics vary from run to run in the last bits of FP64
    assert loss.shape == () and loss.dtype == torch.float32 and abs(loss.item() - value.item()) <= 1e-7 * abs(value.item())
    assert torch.equal(img.grad, 2.0 * grad)
