"""Render walks, per 8x8 quadrant of a tile, only the staged Gaussians that can
reach alpha_low in it: Gaussians much smaller than a quadrant, long and thin
ones that cross its corners, large ones, list lengths around the batch of 256,
images that end inside a quadrant, and low and high alpha_low."""
import numpy as np
import pytest

import oracle
from paper_2409_08669_gb300 import scenes as S
from parity_utils import compare_images, gpu_forward

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _scene(kind, n, rng):
    scene = S.tiny_scene(int(rng.integers(1 << 30)), n=n)
    if kind == "mixed":
        kinds = rng.integers(0, 3, n)
    else:
        kinds = np.full(n, ("specks", "needles", "blobs").index(kind))
    specks = np.exp(rng.normal(-7.0, 0.5, (n, 3)))
    needles = np.exp(rng.normal(-6.0, 0.5, (n, 3)))
    needles[:, 0] = np.exp(rng.normal(-1.5, 0.5, n))
    blobs = np.exp(rng.normal(-1.5, 0.3, (n, 3)))
    scene.scales[:] = np.choose(kinds[:, None], (specks, needles, blobs)).astype(np.float32)
    scene.opac[:] = rng.uniform(0.002, 0.3, n).astype(np.float32)
    return scene


@pytest.mark.parametrize("kind,n,w,h,mode,alpha_low,t_min", [
    ("specks", 3000, 33, 17, "plain", 1 / 255, 1e-4),
    ("needles", 1500, 101, 75, "plain", 1 / 255, 1e-4),
    ("needles", 1500, 101, 75, "aabb", 1e-6, 0.0),
    ("blobs", 255, 40, 72, "aabb", 0.05, 1e-4),
    ("blobs", 256, 40, 72, "plain", 1 / 255, 1e-4),
    ("blobs", 257, 7, 9, "plain", 1 / 255, 0.0),
    ("mixed", 2500, 129, 65, "circle", 1 / 255, 1e-4),
])
def test_quadrant_lists_render_the_oracles_frame(kind, n, w, h, mode, alpha_low, t_min):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2409_08669_gb300.raster import Rasterizer, upload
    rng = np.random.default_rng(n + w)
    scene = _scene(kind, n, rng)
    cam = S.look_at((0.4, 0.3, -3.0), width=w, height=h)
    st = S.Settings(mode={"plain": S.MODE_PLAIN, "circle": S.MODE_CIRCLE, "aabb": S.MODE_AABB}[mode],
                    alpha_low=alpha_low, t_min=t_min)
    rast = Rasterizer(max_gaussians=n, pair_capacity=1 << 20, max_width=w, max_height=h)
    try:
        img, t_final, load = gpu_forward(rast, upload(scene), cam, st)
    finally:
        rast.close()
    ref = oracle.render(scene, cam, st)
    # a Gaussian dropped from a quadrant it reaches changes l_i at a pixel far from
    # every threshold; pixels within tolerance of one may differ, one in a thousand
    compare_images(img, t_final, load, ref, ref["near"] != 0, max_logged_frac=1e-3)
