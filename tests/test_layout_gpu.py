"""The render layouts of a resident volume at their edges: entries of 2^3 voxels in blocks of 2^3,
16-bit ones packed, written in spans of a row: sizes from one voxel up, the whole range
of each type, after an upload and after an update. Images within the suite's 1e-4 of the FP64
oracle; the staged kernel reads another copy of the volume and must agree bit for bit."""
import numpy as np
import pytest

from paper_2005_01442_gb300 import synth

pytestmark = pytest.mark.gpu

TOL = 1e-4


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
@pytest.mark.parametrize("shape", [(1, 1, 1), (1, 2, 3), (3, 1, 2), (2, 5, 4), (6, 7, 8),
                                   (5, 4, 33), (3, 6, 132), (2, 3, 259), (3, 2, 523)])
def test_layouts_of_every_size(R, orc, torch, shape, dtype):
    rng = np.random.default_rng(sum(shape))
    lo, hi = (0.0, 65535.0) if dtype == np.uint16 else (-32768.0, 32767.0)
    tf = synth.tf_random(4, 6)
    tf[:, 3] = 0.02 + 0.2 * tf[:, 3]
    vols = [rng.integers(int(lo), int(hi) + 1, shape).astype(dtype) for _ in range(2)]
    vols[0].flat[0], vols[0].flat[-1] = lo, hi  # the ends of the range, at the corners
    dims = synth.dims_of(vols[0])
    cams = [synth.ortho_z_camera(dims, 9, 7), synth.orbit_cameras(3, 1, dims, 14, 12)[0]]
    vid = R.upload_volume(vols[0])
    tid = R.set_tf(tf, lo, hi)
    for k, vol in enumerate(vols):
        if k:
            R.update_volume(vid, torch.from_numpy(vol).cuda() if dtype != np.uint16 else vol)
        for cam in cams:
            for variant in ({}, {"interp": 1}, {"preclass": 1}, {"interp": 1, "preclass": 1},
                            {"phong": (0.3, 0.7, 0.25, 16.0)}):
                ref = orc.render(vol, tf, lo, hi, cam, 0.5, **variant)
                for kernel in (0, 1):
                    img = R.render(vid, tid, cam, kernel=kernel, **variant).cpu().numpy()
                    assert np.abs(img - ref).max() <= TOL
            staged = R.render(vid, tid, cam, kernel=7)
            assert torch.equal(staged, R.render(vid, tid, cam, kernel=1))
    R.free_tf(tid)
    R.free_volume(vid)
