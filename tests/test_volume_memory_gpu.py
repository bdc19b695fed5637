"""Device memory of a resident volume: the padded copy in the voxel type and 16 bytes a voxel of
render layout, for every voxel type; and the float32 layout's entries at the far face along y,
which odd and even sizes end in different blocks."""
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


@pytest.mark.parametrize("dtype,size", [("int16", 2), ("uint16", 2), ("float32", 4)])
def test_a_volume_takes_16_bytes_a_voxel_and_its_copy(R, torch, dtype, size):
    n = (258, 255, 256)  # z, y, x
    vol = torch.zeros(n, dtype=getattr(torch, dtype), device="cuda")
    padded = (n[0] + 6) * (n[1] + 6) * (n[2] + 12)
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    vid = R.upload_volume(vol)
    used = before - torch.cuda.mem_get_info()[0]
    R.free_volume(vid)
    assert used <= (16 + size) * padded + (8 << 20), used / padded  # (two allocations' granularity)


@pytest.mark.parametrize("shape", [(6, 1, 5), (5, 2, 9), (4, 3, 7), (9, 17, 8), (8, 18, 131)])
def test_float32_samples_up_to_the_far_faces(R, orc, torch, shape):
    vol = np.random.default_rng(7).uniform(0.0, 1000.0, shape).astype(np.float32)
    i = np.arange(256, dtype=np.float32)[:, None] / 255.0
    tf = np.concatenate([i, 1.0 - i, i * i, 0.02 + 0.2 * i], 1).astype(np.float32)
    vid, tid = R.upload_volume(vol), R.set_tf(tf, 0.0, 1000.0)
    dims = synth.dims_of(vol)
    cams = [synth.ortho_z_camera(dims, 24, 24), synth.orbit_cameras(5, 1, dims, 31, 22)[0]]
    for cam in cams:
        for variant in ({}, {"interp": 1}, {"preclass": 1}, {"kernel": 1}):
            img = R.render(vid, tid, cam, step=0.3, **variant).cpu().numpy()
            opts = {k: v for k, v in variant.items() if k != "kernel"}
            ref = orc.render(vol, tf, 0.0, 1000.0, cam, 0.3, **opts)
            assert np.abs(img - ref).max() <= 1e-4  # the suite's bound for images
    R.free_tf(tid)
    R.free_volume(vid)
