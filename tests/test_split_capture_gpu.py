"""Renders captured in graphs: every replay starts from a cleared queue of the graph's own, so
replays on other streams, renders on the stream it was captured on and regrown queues spoil
neither each other's images nor later ones."""
import ctypes as C

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
def scene(torch):
    from paper_2005_01442_gb300 import build
    from paper_2005_01442_gb300.renderer import Renderer
    build.build()
    r = Renderer(0)
    vol = synth.ct_volume((40, 48, 56), seed=3)
    vid = r.upload_volume(vol)
    r.build_bricks(vid, 8)
    tid = r.set_tf(synth.tf_ct(), synth.CT_LO, synth.CT_HI)
    dims = synth.dims_of(vol)
    yield r, vid, tid, [synth.orbit_cameras(k, 1, dims, w, h)[0]
                        for k, (w, h) in enumerate([(160, 120), (157, 93), (320, 240)])]
    r.close()


MEMSET = 2  # CU_GRAPH_NODE_TYPE_MEMSET


def test_a_captured_render_clears_its_queue(scene, torch):
    R, vid, tid, cams = scene
    cu = C.CDLL("libcuda.so.1")
    s = torch.cuda.Stream()
    out = torch.zeros((cams[0].height, cams[0].width, 4), device="cuda")
    R.render(vid, tid, cams[0], brick=8, out=out, stream=s)
    torch.cuda.synchronize()
    ptr, graph, n = C.c_void_p(s.cuda_stream), C.c_void_p(), C.c_size_t()
    assert cu.cuStreamBeginCapture_v2(ptr, 2) == 0  # relaxed
    try:
        R.render(vid, tid, cams[0], brick=8, out=out, stream=s)
    finally:
        assert cu.cuStreamEndCapture(ptr, C.byref(graph)) == 0
    assert cu.cuGraphGetNodes(graph, None, C.byref(n)) == 0
    nodes = (C.c_void_p * n.value)()
    assert cu.cuGraphGetNodes(graph, nodes, C.byref(n)) == 0
    types = []
    for node in nodes:
        t = C.c_int()
        assert cu.cuGraphNodeGetType(C.c_void_p(node), C.byref(t)) == 0
        types.append(t.value)
    cu.cuGraphDestroy(graph)
    assert types.count(MEMSET) == 1 and len(types) == 3, types


def test_replays_beside_renders_on_the_capture_stream(scene, torch):
    R, vid, tid, cams = scene
    want = [R.render(vid, tid, c, brick=8) for c in cams]
    side, other = torch.cuda.Stream(), torch.cuda.Stream()
    images = [torch.zeros_like(w) for w in want]
    with torch.cuda.stream(side):
        R.render(vid, tid, cams[0], brick=8, out=images[0])
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=side):
        R.render(vid, tid, cams[0], brick=8, out=images[0])
    eager = [torch.zeros_like(want[1]) for _ in range(20)]
    got = []
    torch.cuda.synchronize()
    for k in range(20):  # replays on one stream beside renders on the stream of the capture
        with torch.cuda.stream(other):
            graph.replay()
            got.append(images[0].clone())
        R.render(vid, tid, cams[1], brick=8, out=eager[k], stream=side)
    torch.cuda.synchronize()
    assert all(torch.equal(g, want[0]) for g in got)
    assert all(torch.equal(e, want[1]) for e in eager)
    # the stream's queue grows (its old one is freed), then a second, larger graph is captured
    R.render(vid, tid, cams[2], brick=8, out=images[2], stream=side)
    torch.cuda.synchronize()
    assert torch.equal(images[2], want[2])
    larger = torch.cuda.CUDAGraph()
    with torch.cuda.graph(larger, stream=side):
        R.render(vid, tid, cams[2], brick=8, out=images[2])
    for _ in range(3):
        images[0].zero_()
        images[2].zero_()
        graph.replay()
        larger.replay()
        torch.cuda.synchronize()
        assert torch.equal(images[0], want[0]) and torch.equal(images[2], want[2])
    assert R.last_device_error() == 0
