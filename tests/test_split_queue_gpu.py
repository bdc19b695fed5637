"""The split render's queue from one frame to the next: the second phase leaves it empty, whatever
the image sizes that follow one another, on several streams, and captured in a graph."""
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


SIZES = [(1, 1), (33, 7), (160, 120), (8, 4), (161, 119), (64, 64)]


def test_frames_after_one_another(R, torch):
    vol = synth.ct_volume((40, 48, 56), seed=3)
    vid = R.upload_volume(vol)
    R.build_bricks(vid, 8)
    tid = R.set_tf(synth.tf_ct(), synth.CT_LO, synth.CT_HI)
    cams = [synth.orbit_cameras(k, 1, synth.dims_of(vol), w, h)[0] for k, (w, h) in
            enumerate(SIZES)]
    # an image of the split render and its per-ray counterpart composite in another order
    alone = [R.render(vid, tid, c, brick=8, kernel=1) for c in cams]
    first = [R.render(vid, tid, c, brick=8) for c in cams]
    for a, b in zip(alone, first):
        assert float((a - b).abs().max()) <= 1e-3
    streams = [torch.cuda.Stream() for _ in range(3)]
    out = [[torch.empty_like(a) for a in first] for _ in streams]
    torch.cuda.synchronize()
    for _ in range(3):
        for s, images in zip(streams, out):
            with torch.cuda.stream(s):
                for c, o in zip(cams, images):
                    R.render(vid, tid, c, brick=8, out=o)
    torch.cuda.synchronize()
    for images in out:
        for o, a in zip(images, first):
            assert torch.equal(o, a)

    side = torch.cuda.Stream()
    image = torch.zeros_like(first[2])
    with torch.cuda.stream(side):  # the queue of this stream is made before the capture
        R.render(vid, tid, cams[2], brick=8, out=image)
    side.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=side):
        R.render(vid, tid, cams[2], brick=8, out=image)
    for _ in range(3):
        image.zero_()
        graph.replay()
        torch.cuda.synchronize()
        assert torch.equal(image, first[2])
    R.free_tf(tid)
    R.free_volume(vid)
