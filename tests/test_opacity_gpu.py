"""The opacity of one segment, 1 - (1 - a)^delta, and its derivative, over table opacities from 0 to
1 and segment lengths from 0.001 to 3.8, against 64 bits.

A constant 3^3 volume at step 10 is one segment a ray, as long as the ray's way through the box.
Bounds: lg2 errs by 2^-22 (relative where |lg2| > 1) and ex2 by 2^-22 of its result, so the power
p = 2^(delta lg2(1 - a)) errs by p (ln 2 delta max(1, |lg2(1 - a)|) + 1) 2^-22; delta itself by
3e-7 of a voxel at either end; 1 - p rounds by 2^-24."""
import numpy as np
import pytest

from paper_2005_01442_gb300 import synth

pytestmark = pytest.mark.gpu

ALPHAS = [0.0, 1e-40, 1e-20, 3e-8, 1e-7, 1e-5, 1e-3, 0.01, 0.1, 0.3, 0.5, 0.7, 0.9, 0.99, 0.9999,
          1.0 - 2.0 ** -20, 1.0 - 2.0 ** -24, 1.0]


def test_opacity_and_its_derivative(orc):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2005_01442_gb300 import build
    from paper_2005_01442_gb300.renderer import Renderer
    build.build()
    vol = np.full((3, 3, 3), 500.0, np.float32)
    cams = synth.orbit_cameras(3, 3, (3, 3, 3), 40, 32)
    unit = np.float32([0.5, 0.25, 1.0, 0.0])
    with Renderer(0) as R:
        vid = R.upload_volume(vol)
        for a in ALPHAS:
            tf = np.tile(unit, (256, 1))
            tf[:, 3] = a
            tid = R.set_tf(tf, 0.0, 1000.0)
            a64 = min(float(np.float32(a)), 1.0 - 2.0 ** -24)
            half = np.tile(unit, (256, 1))
            half[:, 3] = 0.5
            for cam in cams:
                # lengths from the FP64 oracle at opacity 1/2
                ref = orc.render(vol, half, 0.0, 1000.0, cam, 10.0)[..., 3]
                delta = -np.log2(1.0 - ref)
                assert 3.0 < delta.max() < 5.3 and (delta > 0).mean() > 0.2
                log = np.log2(1.0 - a64)
                p = 2.0 ** (delta * log)
                err = p * (np.log(2) * delta * max(1.0, abs(log)) + 1.0) * 2.0 ** -22
                err += p * np.log(2) * abs(log) * 6e-7 + 2.0 ** -24
                img = R.render(vid, tid, cam, step=10.0).cpu().numpy().astype(np.float64)
                assert (np.abs(img[..., 3] - (1.0 - p)) <= err).all()
                if not 0.0 < np.float32(a) < np.float32(1.0 - 2.0 ** -24):
                    continue  # at its ends the clamp has derivative zero
                g = torch.zeros((cam.height, cam.width, 4), device="cuda")
                g[..., 3] = 1.0
                gtf = torch.zeros((256, 4), device="cuda")
                R.render_backward(vid, tid, cam, g, gtf, None, step=10.0, ert=1.0)
                hit = delta[delta > 0]
                want = hit * (1.0 - a64) ** (hit - 1.0)
                rel = (np.log(2) * np.abs(hit - 1.0) * max(1.0, abs(log)) + 1.0) * 2.0 ** -22
                rel = rel + 6e-7 * (1.0 / hit + np.log(2) * abs(log))
                # the sum over the rays: terms of one sign, each of its sums rounds
                got = float(gtf[:, 3].double().sum())
                assert abs(got - want.sum()) <= (want * rel).sum() + want.sum() * hit.size * 2.0 ** -24
            R.free_tf(tid)
