"""A compressed mesh takes other vertex colours after its upload: its positions
are the context's own encoding, so nothing but the colours is read or changed."""
import numpy as np
import pytest
import torch

import synthetic as S
from synthetic.scenes import Camera, Instance, Scene

from gpu_util import u64, upload

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("first", [False, True])
def test_other_colours(first):
    import __graft_entry__ as g
    g.build()
    from paper_2604_21749_gb300 import api
    W, H = 320, 200
    hf = S.heightfield_mesh(40, seed=6)
    cam = Camera(S.look_at((0.5, 1.2, -0.4), (0.5, 0.0, 0.5)), S.perspective(60.0, W / H, 0.01, 100.0), W, H)
    scene = Scene([hf], [Instance(0, np.eye(4, dtype=np.float32))], [cam])
    colours = torch.flip(hf.rgba8, dims=[0]).contiguous().cuda()
    r = api.Renderer(0)
    keep = upload(r, scene, with_colour=first, compressed=(0,))
    info = r.mesh_info(0)
    before = r.render(cam.view, cam.proj, W, H)
    r.update_mesh(0, rgba8=colours)
    with pytest.raises(api.CurastError):
        r.update_mesh(0, pos=keep[0][0])
    after = r.render(cam.view, cam.proj, W, H)
    image = r.resolve(cam.view, cam.proj, after)
    r.sync()
    assert r.mesh_info(0) == info and (u64(after) == u64(before)).all() and (before != -1).any()
    fresh = api.Renderer(0)
    fresh.upload_mesh(keep[0][0], keep[0][1], colours, compressed=True)
    fresh.add_instance(0)
    want = fresh.resolve(cam.view, cam.proj, fresh.render(cam.view, cam.proj, W, H))
    fresh.sync()
    for a, b in zip(image, want):
        assert torch.equal(a, b)
