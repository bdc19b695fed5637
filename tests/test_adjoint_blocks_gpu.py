"""The adjoint's blocks of 32 samples and boxes of voxel gradients at their edges: segments of 1 to
4 blocks and of a part of one, steps so long that fewer samples share a box, rows of the volume
on and off 16-byte boundaries, volumes thinner than a sample's taps, images of part tiles.

The table is linear in the index, so neither gradient has kinks. Both are sums of contributions of
either sign, which nearly cancel in some entries, so the suite's bound for continuous gradients
(1e-3 of the FP64 oracle's) holds for the norm of the difference and, against the largest, for
each entry and voxel."""
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


def _close(g, ref):
    assert np.abs(ref).max() > 0
    assert np.linalg.norm(g - ref) <= 1e-3 * np.linalg.norm(ref)
    assert np.abs(g - ref).max() <= 1e-3 * np.abs(ref).max()


@pytest.mark.parametrize("shape,image,seg,step", [
    ((44, 36, 40), (37, 29), 64, 0.5),   # rows of 40: float4 atomics
    ((44, 36, 40), (37, 29), 16, 0.37),
    ((44, 36, 40), (37, 29), 48, 0.25),
    ((44, 36, 40), (37, 29), 128, 0.11),
    ((39, 41, 43), (33, 30), 64, 0.5),   # odd rows
    ((30, 90, 61), (31, 17), 64, 1.7),   # fewer samples a box
    ((90, 30, 64), (31, 17), 32, 6.0),   # one sample a box
    ((2, 3, 1), (9, 5), 64, 0.1),
    ((1, 40, 3), (16, 16), 112, 0.2),
    ((20, 22, 24), (300, 240), 64, 0.5),  # tiles of 8 x 4
])
def test_gradients_of_every_block_size(R, orc, torch, shape, image, seg, step):
    rng = np.random.default_rng(sum(shape) + seg)
    vol = rng.uniform(100.0, 900.0, shape).astype(np.float32)
    i = np.arange(256, dtype=np.float64)[:, None] / 255.0
    tf = (np.array([0.9, 0.1, 0.4, 0.002]) * (1 - i) + np.array([0.2, 0.8, 0.5, 0.03]) * i)
    tf = tf.astype(np.float32)
    vid = R.upload_volume(vol)
    tid = R.set_tf(tf, 0.0, 1000.0)
    cam = synth.orbit_cameras(7, 1, synth.dims_of(vol), *image)[0]
    g = rng.normal(0, 1, (cam.height, cam.width, 4)).astype(np.float32)
    g[rng.random(g.shape[:2]) < 0.2] = 0.0  # rays without a gradient
    gtf = torch.zeros((256, 4), device="cuda")
    gvol = torch.zeros(shape, device="cuda")
    R.render_backward(vid, tid, cam, torch.from_numpy(g).cuda(), gtf, gvol, step=step, ert=1.0,
                      brick=0, seg_len=seg)
    rtf, rvol = orc.render_grad(vol, tf, 0.0, 1000.0, cam, step, g.astype(np.float64), ert=1.0,
                                brick=0)
    _close(gtf.cpu().numpy().astype(np.float64), rtf)
    _close(gvol.cpu().numpy().astype(np.float64), rvol)
    only = torch.zeros((256, 4), device="cuda")  # without voxel gradients
    R.render_backward(vid, tid, cam, torch.from_numpy(g).cuda(), only, None, step=step, ert=1.0,
                      brick=0, seg_len=seg)
    _close(only.cpu().numpy().astype(np.float64), rtf)
    R.free_tf(tid)
    R.free_volume(vid)
