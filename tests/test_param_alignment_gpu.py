"""Parameter arrays of 4-byte alignment (slices of larger ones; rots and sh are
16-byte aligned): the same frame as from aligned copies.  More Gaussians than one
wave of Preprocess, whose prefetch of the next wave needs 16 bytes."""
import pytest

from paper_2409_08669_gb300 import scenes as S

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("first", [1, 2, 3])
def test_slices_of_larger_arrays(first):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2409_08669_gb300.raster import Rasterizer, upload
    whole = upload(S.cluster_scene(300_000, seed=4))
    sliced = tuple(p[first:] for p in whole)
    assert sliced[0].data_ptr() % 16 and sliced[3].data_ptr() % 16 and not sliced[2].data_ptr() % 16
    cam, st = S.look_at((4.0, 0.0, 0.5), width=200, height=120), S.Settings(mode=S.MODE_AABB)
    n = sliced[0].shape[0]
    rast = Rasterizer(max_gaussians=n, pair_capacity=1 << 23, max_width=200, max_height=120)
    try:
        want = [t.clone() for t in rast.forward(tuple(p.clone() for p in sliced), cam, st)]
        for w, got in zip(want, rast.forward(sliced, cam, st)):
            assert torch.equal(w, got)
        assert rast.sync_status() == 0 and float(want[2].float().mean()) > 1.0
    finally:
        rast.close()
