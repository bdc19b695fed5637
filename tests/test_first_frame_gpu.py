"""The first frame on a stream, and one whose queue has to grow, make the queue and clear it in the
stream's own order: no stream is created (and none waited for) on the way."""
import ctypes as C

import pytest

from paper_2005_01442_gb300 import synth

pytestmark = pytest.mark.gpu


def test_first_frames_create_no_stream():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2005_01442_gb300 import build
    from paper_2005_01442_gb300.renderer import Renderer
    build.build()
    cu = C.CDLL("libcuda.so.1")

    def stream():
        """A new stream and the number of streams its context has made so far."""
        p, i = C.c_void_p(), C.c_ulonglong()
        assert cu.cuStreamCreate(C.byref(p), 1) == 0  # non-blocking
        assert cu.cuStreamGetId(p, C.byref(i)) == 0
        return torch.cuda.ExternalStream(p.value), p, i.value

    with Renderer(0) as R:
        vol = synth.ct_volume((40, 48, 56), seed=3)
        vid = R.upload_volume(vol)
        R.build_bricks(vid, 8)
        tid = R.set_tf(synth.tf_ct(), synth.CT_LO, synth.CT_HI)
        cams = [synth.orbit_cameras(k, 1, synth.dims_of(vol), w, h)[0]
                for k, (w, h) in enumerate([(64, 48), (200, 150)])]
        want = [R.render(vid, tid, c, brick=8) for c in cams]
        out = [torch.zeros_like(w) for w in want]
        torch.cuda.synchronize()
        made = [stream()]
        for k in range(3):  # streams made one after the other, with renders between the last two
            if k == 1:
                for c, o in zip(cams, out):  # a new queue, then a larger one
                    R.render(vid, tid, c, brick=8, out=o, stream=made[0][0])
            made.append(stream())
        torch.cuda.synchronize()
        ids = [i for _, _, i in made]
        assert ids[2] - ids[1] == ids[1] - ids[0] == ids[3] - ids[2], ids
        assert all(torch.equal(o, w) for o, w in zip(out, want))
        for _, p, _ in made:
            assert cu.cuStreamDestroy_v2(p) == 0
