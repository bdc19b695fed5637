"""Leaping over 8^3 tiles in renders with bricks of 16, and the distance fields over rows of a
multiple of four bricks and not: skipping changes no bit of an image, whatever the sizes, types
and variants, and counting samples changes neither image nor the bricks that are counted."""
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


@pytest.mark.parametrize("dtype", [np.uint16, np.int16, np.float32])
@pytest.mark.parametrize("shape", [(1, 1, 1), (8, 9, 7), (16, 17, 33), (40, 24, 96), (100, 70, 33),
                                   (130, 50, 256), (61, 203, 120)])
def test_skipping_changes_no_bit(R, orc, torch, shape, dtype):
    rng = np.random.default_rng(sum(shape))
    vol = np.where(rng.random(shape) < 0.0007, 900, 30).astype(dtype)
    vol.flat[0] = vol.flat[-1] = 900
    tf = synth.tf_ct()
    lo, hi = synth.CT_LO, synth.CT_HI
    vid = R.upload_volume(vol)
    tid = R.set_tf(tf, lo, hi)
    for B in (8, 16):
        R.build_bricks(vid, B)
    dims = synth.dims_of(vol)
    cams = [synth.ortho_z_camera(dims, 21, 19)] + synth.orbit_cameras(sum(shape), 4, dims, 50, 39)
    for k, cam in enumerate(cams):
        for variant in ({}, {"interp": 1}, {"phong": (0.3, 0.7, 0.25, 16.0)}):
            for kernel in (0, 1):
                none = R.render(vid, tid, cam, brick=0, kernel=kernel, **variant)
                for B in (8, 16):
                    img = R.render(vid, tid, cam, brick=B, kernel=kernel, **variant)
                    assert torch.equal(img, none)
        cnt = torch.zeros(3, dtype=torch.int64, device="cuda")
        img = R.render(vid, tid, cam, brick=16, counters=cnt, ert=1.0)
        assert torch.equal(img, R.render(vid, tid, cam, brick=16, ert=1.0))
        if k == 0:
            _, counts = orc.render(vol, tf, lo, hi, cam, 0.5, ert=1.0, brick=16,
                                   return_counts=True)
            assert cnt.tolist()[:2] == [int(c) for c in counts[:2]]
    R.free_tf(tid)
    R.free_volume(vid)
