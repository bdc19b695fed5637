"""The occupancy structures of a (volume, transfer function): the cell mask at the edges of its
tiles and blocks, and leaping fields longer than their cap, against the FP64 oracle. All
decisions are exact (tables equal byte for byte, images equal bit for bit)."""
import numpy as np
import pytest

from paper_2005_01442_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return torch


@pytest.fixture(scope="module")
def R(torch):
    from paper_2005_01442_gb300 import build
    from paper_2005_01442_gb300.renderer import Renderer
    build.build()
    r = Renderer(0)
    yield r
    r.close()


@pytest.mark.parametrize("B", [8, 16])
@pytest.mark.parametrize("dtype", [np.uint16, np.int16, np.float32])
@pytest.mark.parametrize("shape", [(1, 1, 1), (2, 3, 5), (7, 8, 9), (15, 16, 17), (4, 31, 63),
                                   (33, 12, 68), (9, 7, 130)])
def test_cell_mask_at_tile_edges(R, orc, shape, dtype, B):
    """Sizes on either side of the mask's blocks (4), tiles (8), bricks and rows of tiles (64);
    sparse values, so that some tiles hold occupied bricks and some none."""
    rng = np.random.default_rng(sum(shape) + B)
    vol = np.where(rng.random(shape) < 0.004, 900, 30).astype(dtype)
    vol.flat[-1] = 900  # the last cell of every axis is open
    tf = synth.tf_ct()
    vid = R.upload_volume(vol)
    R.build_bricks(vid, B)
    tid = R.set_tf(tf, synth.CT_LO, synth.CT_HI)
    assert np.array_equal(R.cellmask(vid, tid, B), orc.cellmask(vol, tf, synth.CT_LO, synth.CT_HI))
    R.free_tf(tid)
    R.free_volume(vid)


@pytest.mark.parametrize("axis", [0, 1, 2])
def test_leaps_longer_than_the_field_cap(R, orc, torch, axis):
    """A volume of 270 bricks along one axis with visible voxels only near its ends: distances
    reach their cap of 255 bricks in both directions."""
    shape = [10, 10, 10]
    shape[axis] = 2160
    vol = np.full(shape, -1000, np.int16)
    np.moveaxis(vol, axis, 0)[3:6, 4:7, 4:7] = 1000
    np.moveaxis(vol, axis, 0)[-4:-2, 2:5, 5:8] = 1000
    dims = synth.dims_of(vol)
    vid = R.upload_volume(vol)
    R.build_bricks(vid, 8)
    tf = synth.tf_ct()
    tid = R.set_tf(tf, synth.CT_LO, synth.CT_HI)
    world = 2 - axis  # array axis -> coordinate
    for sign in (-1.0, 1.0):
        eye = [4.1, 4.3, 4.7]
        eye[world] = 1080.0 + sign * 1600.0
        center = [4.5, 4.5, 4.5]
        center[world] = 1080.0
        up = (0.0, 0.0, 1.0) if world == 1 else (0.0, 1.0, 0.0)
        cam = synth.Camera(1, tuple(eye), tuple(center), up, 0.0, (14.0, 14.0), 20, 18).as_float32()
        ref = orc.render(vol, tf, synth.CT_LO, synth.CT_HI, cam, 0.5, brick=8)
        counts = []
        assert dims[world] == 2160 and ref[..., 3].max() > 0.5
        for kernel in (0, 1):
            cnt = torch.zeros(3, dtype=torch.int64, device="cuda")
            img = R.render(vid, tid, cam, brick=8, kernel=kernel, counters=cnt)
            none = R.render(vid, tid, cam, brick=0, kernel=kernel)
            assert torch.equal(img, none)
            assert torch.equal(R.render(vid, tid, cam, brick=8, kernel=kernel), none)
            assert abs(img.cpu().numpy() - ref).max() <= 1e-4
            counts.append(cnt.tolist()[:2])
        # two marching codes, the same samples in occupied bricks. (The oracle counts one more
        # sample on some rays: these are 2160 voxels and 1e-4 long, 4321 segments in float64
        # and 4320 in float32, where the last one is lost in rounding.)
        assert counts[0] == counts[1] and counts[0][1] > 0
    R.free_tf(tid)
    R.free_volume(vid)
