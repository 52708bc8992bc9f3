"""The screen passes of a large image with more than 64 triangles a pixel walk one
row a thread, with fewer four: the same image either way."""
import pytest
import torch

import synthetic as S
from synthetic.scenes import Camera, Instance, Scene

from gpu_util import upload

pytestmark = pytest.mark.gpu


def test_images_do_not_depend_on_the_density():
    """A mesh alone, and beside the 300 million triangles of instances out of
    sight, at 2003 x 2001 pixels."""
    import __graft_entry__ as g
    import numpy as np
    g.build()
    from paper_2604_21749_gb300 import api
    W, H = 2003, 2001
    hf, big = S.heightfield_mesh(300, seed=4), S.heightfield_mesh(1500, seed=5)
    uv, tex = S.grid_uv(300).cuda(), S.texture_mip_chain(7, seed=1).cuda()
    cam = Camera(S.look_at((0.5, 1.2, -0.4), (0.5, 0.0, 0.5)), S.perspective(60.0, W / H, 0.01, 100.0), W, H)
    away = np.eye(4, dtype=np.float32)
    away[2, 3] = -500.0
    out = []
    for others in (0, 70):
        assert (2 * 300 ** 2 + others * 2 * 1500 ** 2 >= 64 * W * H) == (others > 0)
        sc = Scene([hf, big], [Instance(0, np.eye(4, dtype=np.float32))] + [Instance(1, away)] * others, [cam])
        r = api.Renderer(0)
        keep = upload(r, sc)
        r.set_mesh_texture(0, uv, tex, 7)
        vis = r.render(cam.view, cam.proj, W, H)
        attr = torch.rand((hf.V, 3), generator=torch.Generator().manual_seed(1)).cuda()
        out.append([vis, *r.resolve(cam.view, cam.proj, vis), *r.resolve_textured(cam.view, cam.proj, vis),
                    r.interpolate(0, cam.view, cam.proj, vis, attr)])
        r.sync()
        r.close()
        del keep
    assert (out[0][0] != -1).any()
    for a, b in zip(*out):
        assert torch.equal(a, b)
