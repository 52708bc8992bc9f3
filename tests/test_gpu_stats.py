"""The counters of curast_sync: every (triangle, pair) that enters stage 1 is
counted in one class, and the classes are what include/curast.h calls them."""
import numpy as np
import pytest
import torch

import synthetic as S
from oracle import oracle as orc
from synthetic.scenes import Camera, Instance, Mesh, Scene
from test_cull_bounds import _exact

from gpu_util import upload
from test_gpu_stage1_exact import _slivers

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def api():
    import __graft_entry__ as g
    g.build()
    from paper_2604_21749_gb300 import api as A
    return A


def _stats(api, scene, **config):
    cam = scene.cameras[0]
    r = api.Renderer(0)
    r.set_config(collect_stats=1, **config)
    keep = upload(r, scene, with_colour=False)
    r.render(cam.view, cam.proj, cam.W, cam.H)
    st = r.sync()
    del keep
    assert st["triangles_in"] == (st["culled_clip"] + st["culled_backface"] + st["culled_tiny"] + st["stage1_rasterized"] +
                                  st["queued_stage2"]), st
    return st


@pytest.mark.parametrize("group", [0, 2])
@pytest.mark.parametrize("copies", [1, 3])
@pytest.mark.parametrize("order", ["rows", "shuffled"])
def test_back_faces_and_tiny_triangles(api, order, copies, group):
    """Closed surfaces, whole on the screen, of triangles larger and smaller than a
    pixel: what is dropped for its facing is counted under that name, with and
    without the conservative cull."""
    fine, coarse = S.sphere_mesh(90, seed=2), S.sphere_mesh(14, seed=3)
    if order == "shuffled":
        fine, coarse = (Mesh(pos=m.pos, idx=m.idx[torch.from_numpy(np.random.default_rng(1).permutation(m.T))].contiguous())
                        for m in (fine, coarse))
    W, H = 480, 270
    cam = Camera(S.look_at((0.0, 0.3, 6.0), (0.0, 0.0, 0.0)), S.perspective(60.0, W / H, 0.1, 50.0), W, H)
    inst = []
    for k in range(2 * copies):
        m = np.diag([0.7, 0.7, 0.7, 1.0]).astype(np.float32)
        m[:3, 3] = (2.0 * (k % 3) - 2.0, 0.9 - 1.8 * (k // 3), 0.0)
        inst.append(Instance(k % 2, m))
    scene = Scene([fine, coarse], inst, [cam])
    cp = orc.camera_params(np.asarray(cam.proj, np.float32))
    back = none = both = 0
    for it in inst:
        mesh = scene.meshes[it.mesh]
        pts = mesh.pos.numpy()[mesh.idx.numpy().astype(np.int64)]
        X, Y, inside = _exact(orc.model_view(np.asarray(cam.view, np.float32), it.model), cp, cam, pts)
        assert inside.all()
        X, Y = (np.rint(256 * v + 128).astype(np.int64) for v in (X, Y))
        area = (X[:, 1] - X[:, 0]) * (Y[:, 2] - Y[:, 0]) - (X[:, 2] - X[:, 0]) * (Y[:, 1] - Y[:, 0])
        empty = (-((128 - X.min(1)) >> 8) > (X.max(1) - 128) >> 8) | (-((128 - Y.min(1)) >> 8) > (Y.max(1) - 128) >> 8)
        back += int((area <= 0).sum())
        none += int(empty.sum())
        both += int(((area <= 0) & empty).sum())
    assert back - both > 500 and none - both > 100
    for exact_all in (0, 1):
        st = _stats(api, scene, stage1_group_min_pairs=group, stage1_exact_all=exact_all)
        assert st["culled_clip"] == 0 and st["triangles_in"] == sum(scene.meshes[it.mesh].T for it in inst)
        assert st["culled_backface"] + st["culled_tiny"] == back + none - both
        assert back - both <= st["culled_backface"] <= back, (st, back, both)
        assert none - both <= st["culled_tiny"] <= none, (st, none, both)


HEAVY = [(32, 32), (31, 33), (1024, 1), (40, 25)]


def test_handed_over_triangles_are_counted_once(api):
    """Batches of up to 96 x 1024 pixels, part of which stage 1 hands to stage 2:
    each triangle is stage 1's or stage 2's."""
    st = _stats(api, _slivers(700, 1100, 1060, seed=5, shapes=HEAVY), stage1_max_pixels=1024, stage1_exact_all=1)
    assert st["queue1_overflow"] == 0 and st["stage1_rasterized"] > 0 and st["queued_stage3"] == 0
    assert st["stage2_rasterized"] == st["queued_stage2"] > 100, st


@pytest.mark.parametrize("capacity", [1, 50, 300])
def test_hand_over_to_a_full_queue_is_an_overflow(api, capacity):
    """What the first queue has no room for is rasterized in place and counted as
    that, wherever it was to be queued from; the rest is stage 2's."""
    st = _stats(api, _slivers(700, 1100, 1060, seed=5, shapes=HEAVY), stage1_max_pixels=1024, stage1_exact_all=1,
                queue1_capacity=capacity)
    assert st["queue1_overflow"] == st["queued_stage2"] - capacity > 0, st
    assert st["stage2_rasterized"] == capacity and st["queued_stage3"] == 0, st
