"""Bricks of 16 leap over the bricks or over 8^3 tiles, by the kernel, the image and the volume: the
image is the one without leaping, bit for bit, on either side of each line of that rule."""
import pytest

from paper_2005_01442_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def R():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2005_01442_gb300 import build
    from paper_2005_01442_gb300.renderer import Renderer
    build.build()
    r = Renderer(0)
    yield r
    r.close()


@pytest.mark.parametrize("bricks", [(7, 3, 6), (8, 4, 4), (26, 25, 26)])  # 126, 128, 16900
@pytest.mark.parametrize("image", [(255, 257), (256, 256)])  # 64 Ki pixels less one, 64 Ki
def test_images_on_either_side_of_the_rule(R, bricks, image):
    import torch
    shape = tuple(16 * b - 5 for b in bricks)
    vol = synth.ct_volume(shape, seed=5) if bricks[0] < 20 else None
    if vol is None:  # a large volume of few features, made quickly
        t = torch.full(shape, -1000, dtype=torch.int16, device="cuda")
        t[100:180, 37:300, 120:140] = 300
        t[17:20, 200:203, 3:390] = 1200
        vol = t
    vid = R.upload_volume(vol)
    R.build_bricks(vid, 16)
    tid = R.set_tf(synth.tf_ct(), synth.CT_LO, synth.CT_HI)
    cam = synth.orbit_cameras(11, 1, shape[::-1], *image)[0]
    visible = 0.0
    for kernel in (0, 1, 2, 3, 4, 5, 7):
        plain = R.render(vid, tid, cam, ert=0.999, brick=0, kernel=kernel)
        assert torch.equal(R.render(vid, tid, cam, ert=0.999, brick=16, kernel=kernel), plain)
        visible = max(visible, float(plain.max()))
    assert visible > 0.1
    R.free_tf(tid)
    R.free_volume(vid)
