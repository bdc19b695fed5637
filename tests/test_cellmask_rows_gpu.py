"""Cell masks of volumes of different sizes after one another share the context's buffer of rows."""
import numpy as np
import pytest

from paper_2005_01442_gb300 import synth

pytestmark = pytest.mark.gpu


def test_masks_of_growing_and_shrinking_volumes(orc):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2005_01442_gb300 import build
    from paper_2005_01442_gb300.renderer import Renderer
    build.build()
    with Renderer(0) as R:
        tf = synth.tf_ct()
        tid = R.set_tf(tf, synth.CT_LO, synth.CT_HI)
        vols = [synth.ct_volume(s, seed=3) for s in [(20, 24, 31), (41, 39, 66), (9, 17, 33)]]
        vids = [R.upload_volume(v) for v in vols]
        want = [orc.cellmask(v, tf, synth.CT_LO, synth.CT_HI) for v in vols]
        for vid in vids:
            R.build_bricks(vid, 8)
        for k in (0, 1, 2, 0, 1):
            assert np.array_equal(R.cellmask(vids[k], tid, 8), want[k])
