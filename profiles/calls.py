"""The calls whose kernels the profiles of this folder describe, each once warm and once between
cudaProfilerStart and cudaProfilerStop.

    python profiles/calls.py [CALL ...]      # default: all

Run it under `ncu --profile-from-start off`; by itself it prints nothing and exits 0.
"""
import os
import sys

import numpy as np
import torch

sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))
from paper_2005_01442_gb300 import synth  # noqa: E402
from paper_2005_01442_gb300.renderer import Renderer  # noqa: E402


def main(names):
    R = Renderer(0)
    calls = {}
    vol = synth.ct_volume()  # 512 x 512 x 400 int16
    dims = synth.dims_of(vol)
    data = torch.from_numpy(vol).cuda()
    vid = R.upload_volume(data)
    R.build_bricks(vid, 8)
    ct = R.set_tf(synth.tf_ct(), synth.CT_LO, synth.CT_HI)
    dense = R.set_tf(synth.tf_ct_dense(), synth.CT_LO, synth.CT_HI)
    cam = synth.orbit_cameras(4, 1, dims, 1024, 1024)[0]
    out = torch.empty((1024, 1024, 4), device="cuda")

    def rebuild():
        R.build_bricks(vid, 8)
        R.build_occupancy(vid, ct, 8)

    def rebuild16():
        R.build_bricks(vid, 16)
        R.build_occupancy(vid, ct, 16)

    calls["update"] = lambda: R.update_volume(vid, data)
    calls["rebuild"] = rebuild
    calls["rebuild16"] = rebuild16
    calls["frame"] = lambda: R.render(vid, ct, cam, ert=0.999, brick=8, out=out)
    calls["frame16"] = lambda: R.render(vid, ct, cam, ert=0.999, brick=16, out=out)
    calls["dense"] = lambda: R.render(vid, dense, cam, ert=0.999, brick=8, out=out)
    calls["staged"] = lambda: R.render(vid, dense, cam, ert=0.999, brick=8, out=out, kernel=7)

    def pieces():
        plan = R.build_pieces(vid, ct, 8, (2, 2, 2))
        R.render_sortlast(plan, cam, ert=0.999, out=out)
        R.free_pieces(plan)

    calls["pieces"] = pieces

    # the differentiation workload: 256^3 float32, one 512^2 view, with either table
    half = synth.ct_volume((512, 512, 512), seed=7).astype(np.float32)
    half = half.reshape(256, 2, 256, 2, 256, 2).mean((1, 3, 5))
    fid = R.upload_volume(half)
    R.build_bricks(fid, 8)
    view = synth.orbit_cameras(7, 1, (256, 256, 256), 512, 512)[0]
    g = torch.rand((512, 512, 4), device="cuda") - 0.5
    gtf, gvol = torch.zeros((256, 4), device="cuda"), torch.zeros((256, 256, 256), device="cuda")
    for name, tid in (("train", ct), ("train_dense", dense)):
        ck = R.ckpt_buffer(fid, view, 0.5, 64)

        def step(tid=tid, ck=ck):
            R.render(fid, tid, view, brick=8, ckpt=ck)
            R.render_backward(fid, tid, view, g, gtf, gvol, brick=8, ckpt=ck)
        calls[name] = step

    for name in names or calls:
        calls[name]()
        calls[name]()
        torch.cuda.synchronize()
        torch.cuda.profiler.start()
        calls[name]()
        torch.cuda.synchronize()
        torch.cuda.profiler.stop()


if __name__ == "__main__":
    main(sys.argv[1:])
