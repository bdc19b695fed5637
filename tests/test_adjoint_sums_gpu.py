"""How coarse the sums are that the adjoint adds to the table gradient: each CTA's go to the same
floats, so the fewer rays a sum holds, the more of them are rounded away.

Every ray of an orthographic view of a constant volume contributes the same c to a table entry.
The gradient buffer starts at V = 2^24, where floats are 2 apart: a sum s is lost when s < 1 and
counts when s > 1. With c = 1/48 the sums of n rays are n/48, so they count where n >= 64 (1.33)
and are lost where n <= 32 (0.67); neither is near 1."""
import numpy as np
import pytest

from paper_2005_01442_gb300 import synth

pytestmark = pytest.mark.gpu


def test_sums_of_large_images_hold_64_rays():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2005_01442_gb300 import build
    from paper_2005_01442_gb300.renderer import Renderer
    build.build()
    vol = np.full((8, 8, 8), 100.5, np.float32)
    tf = np.tile(np.array([0.5, 0.5, 0.5, 0.01], np.float32), (256, 1))
    with Renderer(0) as R:
        vid, tid = R.upload_volume(vol), R.set_tf(tf, 0.0, 255.0)

        def gradient(w, h, g, start):
            cam = synth.ortho_z_camera(synth.dims_of(vol), w, h)
            go = torch.zeros((h, w, 4), device="cuda")
            go[..., 0] = g
            out = torch.full((256, 4), start, device="cuda")
            R.render_backward(vid, tid, cam, go, out, None, step=1.0, ert=1.0, brick=0)
            return out.cpu().numpy()[:, 0].astype(np.float64)

        one = gradient(16, 16, 1.0, 0.0)
        assert np.flatnonzero(one).tolist() == [100, 101]
        c = one[100] / 256.0
        w, h = 1448, 1456  # 2.01 Mi pixels, whole tiles of 8 x 8
        got = gradient(w, h, 1.0 / 48.0 / c, 2.0 ** 24)[100] - 2.0 ** 24
        # each sum of 64 rays, 4/3, rounds to 2
        assert got >= 0.99 * 2.0 * (w * h / 64), got
