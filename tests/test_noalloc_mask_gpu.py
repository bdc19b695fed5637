"""vrc_render_noalloc skips clear cells wherever the mask fits behind what the leaping fields need:
4 bytes a brick while they are built. Elsewhere it renders the same image, resampling every sample
of an occupied brick."""
import ctypes as C

import pytest

from paper_2005_01442_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,fits", [((2360, 2048, 8), True), ((2500, 2048, 8), False)])
def test_the_mask_goes_right_behind_the_fields(n, fits):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2005_01442_gb300 import build, native
    from paper_2005_01442_gb300.renderer import Renderer
    build.build()
    up = lambda b: -(-b // 256) * 256  # noqa: E731
    nb = [-(-k // 8) for k in n]
    bricks = nb[0] * nb[1] * nb[2]
    blocks = 1
    for k in n:
        blocks *= (k + 3) // 4 + 1
    fields = up(bricks) + up(8 * bricks)
    corners = (nb[0] + 1) * (nb[1] + 1) * (nb[2] + 1)
    # 8 bytes a block of the mask; 4 bytes a brick leave room for it where 4 per corner would not
    assert (fields + up(4 * bricks) + 8 * blocks <= 8 << 20) == fits
    assert fields + up(4 * corners) + 8 * blocks > 8 << 20
    vol = torch.full(n[::-1], -1000, dtype=torch.int16, device="cuda")
    vol[2:5, 100:110, 100:120] = 300
    with Renderer(0) as R:
        vid = R.upload_volume(vol)
        R.build_bricks(vid, 8)
        tid = R.set_tf(synth.tf_ct(), synth.CT_LO, synth.CT_HI)
        cam = synth.ortho_z_camera(n, 236, 205)
        counts = [torch.zeros(3, dtype=torch.int64, device="cuda") for _ in range(2)]
        want = R.render(vid, tid, cam, ert=0.999, brick=8, kernel=1, counters=counts[0])
        out = torch.empty_like(want)
        native.check(R.ctx, R.lib.vrc_render_noalloc(
            R.ctx, vid, tid, C.byref(native.camera_struct(cam)),
            C.byref(native.params_struct(0.5, 0.999, 8, 64, 1)), C.c_void_p(out.data_ptr()),
            C.c_void_p(counts[1].data_ptr()),
            C.c_void_p(int(torch.cuda.current_stream().cuda_stream))))
        torch.cuda.synchronize()
        assert torch.equal(out, want) and float(want.max()) > 0
        (_, ex0, re0), (_, ex1, re1) = [c.tolist() for c in counts]
        assert 0 < re0 < ex0 == ex1  # clear cells are counted as executed
        assert re1 == (re0 if fits else ex1)
