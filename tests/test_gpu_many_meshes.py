"""Scenes of very many meshes of one instance each: the exact kernel finds the
segment of a bitmap word without walking all of them."""
import numpy as np
import pytest
import torch

import synthetic as S
from synthetic.scenes import Camera, Instance, Mesh, Scene

from gpu_util import assert_vis_equal, oracle_vis, upload

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def api():
    import __graft_entry__ as g
    g.build()
    from paper_2604_21749_gb300 import api as A
    return A


def _instances(n, meshes):
    side = int(np.ceil(np.sqrt(n)))
    out = []
    for k in range(n):
        m = np.eye(4, dtype=np.float32)
        m[0, 3], m[2, 3] = k % side, k // side
        out.append(Instance(k % meshes, m))
    cam = Camera(S.look_at((side / 2, 0.5 * side, -0.2 * side), (side / 2, 0.0, side / 2)),
                 S.perspective(55.0, 1.5, 1e-2, 10.0 * side), 240, 160)
    return out, cam


def test_words_of_many_meshes(api):
    """Meshes of one triangle to three work items, some invisible, so that a
    lane's next word lies one, several or very many segments on."""
    rng = np.random.default_rng(8)
    sizes = [1, 2, 23, 3, 40, 1, 1, 31]
    meshes = [S.heightfield_mesh(n, seed=n) for n in sizes]
    inst, cam = _instances(1500, 1500)
    every = [meshes[int(rng.integers(len(meshes)))] for _ in range(1500)]
    scene = Scene(every, inst, [cam])
    for per_pair in (64, 1):
        r = api.Renderer(0)
        r.set_config(pairs_per_segment=per_pair)
        keep = upload(r, scene, with_colour=False)
        vis = r.render(cam.view, cam.proj, cam.W, cam.H)
        r.sync()
        assert_vis_equal(vis, oracle_vis(scene, cam), f"{per_pair} pairs a segment")
        del keep


def test_many_meshes_cost_little_more_than_many_instances(api):
    """20,000 meshes of one instance against 50 meshes of 400: the same triangles,
    so much the same work in the exact kernel (ten times as long is far beyond
    the difference, and a walk over the segments 58 times)."""
    hf = S.heightfield_mesh(24, seed=2)
    pos, idx = hf.pos.cuda(), hf.idx.cuda()
    best = []
    for count in (50, 20000):
        inst, cam = _instances(20000, count)
        r = api.Renderer(0)
        for _ in range(count):
            r.upload_mesh(pos, idx)
        for it in inst:
            r.add_instance(it.mesh, it.model)
        times = []
        for _ in range(8):
            r.render(cam.view, cam.proj, 1920, 1080)
            r.sync()
            times.append(r.stage_times()[2])
        best.append(min(times))
        r.close()
    assert best[1] < 10 * best[0], best
