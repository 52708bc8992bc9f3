"""The differentiable step's gradients for every number of channels it takes,
each set of gradients wanted, in fresh processes: the backward's block holds
256 rows of gradients in shared memory, and what a launch may use must not
depend on the calls before it."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

# the two calls whose rows just fit 48 KB without the kernel's fixed arrays
FIRST = [(12, "both"), (15, "attr")]


@pytest.mark.parametrize("C,want", FIRST)
def test_every_channel_count(C, want):
    p = subprocess.run([sys.executable, os.path.abspath(__file__), str(C), want], capture_output=True, text=True, timeout=600)
    assert p.returncode == 0, p.stdout[-2000:] + p.stderr[-2000:]


def _gradients(C, want):
    import numpy as np
    import torch

    import synthetic as S
    from gpu_util import u64, upload
    from oracle import adjoint as A
    from oracle import oracle as orc
    from paper_2604_21749_gb300 import api
    from synthetic.scenes import Camera, Instance, Scene
    W, H = 61, 43
    hf = S.heightfield_mesh(20, seed=31)
    cam = Camera(S.look_at((0.5, 1.1, -0.25), (0.5, 0.0, 0.55)), S.perspective(55.0, W / H, 1e-2, 100.0), W, H)
    rng = np.random.default_rng(C)
    attr = rng.uniform(-1, 1, size=(hf.V, C)).astype(np.float32)
    g = rng.normal(size=(H, W, C)).astype(np.float32)
    r = api.Renderer(0)
    keep = upload(r, Scene([hf], [Instance(0, np.eye(4, dtype=np.float32))], [cam]), with_colour=False)
    vis = r.render(cam.view, cam.proj, W, H)
    ga, gp = r.interpolate_backward(0, cam.view, cam.proj, vis, torch.from_numpy(attr).cuda(), torch.from_numpy(g).cuda(),
                                    want_attr=want != "pos", want_pos=want != "attr")
    r.sync()
    fx, fy, _ = orc.camera_params(cam.proj)
    mv = orc.model_view(cam.view, np.eye(4, dtype=np.float32))
    tri = A.pixel_triangles(u64(vis), 0, hf.T)
    da, dp = A.adjoint64(hf.pos.numpy(), hf.idx.numpy(), attr, mv, fx, fy, W, H, tri, g.astype(np.float64).reshape(-1, C))
    for got, ref in ((ga, da), (gp, dp)):
        if got is not None:
            assert np.linalg.norm(got.cpu().numpy() - ref) <= 1e-4 * np.linalg.norm(ref), (C, want)
    del keep


if __name__ == "__main__":
    here = os.path.dirname(os.path.abspath(__file__))
    sys.path[:0] = [here, os.path.dirname(here)]
    import __graft_entry__
    __graft_entry__.build()
    _gradients(int(sys.argv[1]), sys.argv[2])
    for channels in range(1, 17):
        for which in ("attr", "both", "pos"):
            _gradients(channels, which)
