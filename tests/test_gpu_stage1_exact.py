"""The exact kernel of stage 1 at the edges of its pixel loop and of its deal
of the survivor bitmap, and stages 2 and 3 behind it, against the oracle
(bit-exact words)."""
import numpy as np
import pytest
import torch

import synthetic as S
from oracle import oracle as orc
from synthetic.scenes import Camera, Instance, Mesh, Scene

from gpu_util import assert_vis_equal, oracle_vis, upload

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def api():
    import __graft_entry__ as g
    g.build()
    from paper_2604_21749_gb300 import api as A
    return A


SHAPES = [(1, 1), (2, 1), (1, 3), (31, 1), (32, 1), (33, 2), (8, 16), (32, 32), (1024, 1), (1, 1024), (341, 3), (64, 16)]


def _slivers(n, W, H, seed, shapes=SHAPES):
    """Triangles in the plane z = -1 of a camera at the origin whose pixel boxes
    are 1 x 1 .. 1024 x 1, 1 x 1024 and 32 x 32 pixels, some across the border."""
    rng = np.random.default_rng(seed)
    pos = []
    for k in range(n):
        w, h = shapes[k % len(shapes)]
        x, y = rng.uniform(-w / 2, W - w / 2), rng.uniform(-h / 2, H - h / 2)
        p = np.array([[x, y], [x + w, y + rng.uniform(0, h)], [x + rng.uniform(0, w), y + h]])
        z = -1.0 - 0.001 * rng.integers(0, 50)          # layers, several triangles on the same one
        ndc = p / (W, H) * 2 - 1
        pos += [[-z * q[0], -z * q[1], z] for q in ndc]  # the 90 degree camera below: x_clip = x, w = -z
    idx = np.arange(3 * n, dtype=np.int32).reshape(n, 3)
    return Scene([Mesh(pos=torch.tensor(np.array(pos, np.float32)), idx=torch.from_numpy(idx))],
                 [Instance(0, np.eye(4, dtype=np.float32))],
                 [Camera(np.eye(4, dtype=np.float32), S.perspective(90.0, 1.0, 1e-2, 10.0), W, H)])


@pytest.mark.parametrize("limit", [1, 128, 1024])
@pytest.mark.parametrize("n", [1, 95, 96, 97, 700])
def test_pixel_ranges_of_every_shape(api, n, limit):
    """One batch and its neighbours (96 survivors), ranges of 1 .. 1024 pixels
    beside one another, more pixels than one segment of the pixel loop."""
    scene = _slivers(n, 1100, 1060, seed=n)
    cam = scene.cameras[0]
    r = api.Renderer(0)
    r.set_config(stage1_max_pixels=limit, stage1_exact_all=1)
    keep = upload(r, scene, with_colour=False)
    vis = r.render(cam.view, cam.proj, cam.W, cam.H)
    r.sync()
    assert_vis_equal(vis, oracle_vis(scene, cam), f"{n} triangles, limit {limit}")
    del keep


@pytest.mark.parametrize("n", [1, 4, 181, 900, 2200])
def test_bitmap_deal(api, n):
    """Bitmaps dealt out by single words, by 16-byte loads and by runs (8 to
    302,000 words), the camera close enough for dense clusters of survivors."""
    hf = S.heightfield_mesh(n, seed=40 + n)
    W, H = 640, 360
    cam = Camera(S.look_at((0.5, 0.45, 0.2), (0.5, 0.1, 0.55)), S.perspective(60.0, W / H, 1e-3, 100.0), W, H)
    scene = Scene([hf], [Instance(0, np.eye(4, dtype=np.float32))], [cam])
    r = api.Renderer(0)
    keep = upload(r, scene, with_colour=False)
    vis = r.render(cam.view, cam.proj, W, H)
    r.sync()
    assert_vis_equal(vis, oracle_vis(scene, cam), f"{n} x {n} cells")
    del keep


@pytest.mark.parametrize("capacity", [1, 50, 1 << 20])
def test_heavy_batches_are_handed_over(api, capacity):
    """Batches of up to 96 x 1024 pixels: what stage 1 hands to stage 2, and what
    queue 1 has no room for, lands in the buffer all the same."""
    scene = _slivers(700, 1100, 1060, seed=5, shapes=[(32, 32), (31, 33), (1024, 1), (40, 25)])
    cam = scene.cameras[0]
    r = api.Renderer(0)
    r.set_config(stage1_max_pixels=1024, stage1_exact_all=1, queue1_capacity=capacity)
    keep = upload(r, scene, with_colour=False)
    vis = r.render(cam.view, cam.proj, cam.W, cam.H)
    st = r.sync()
    assert st["queued_stage2"] > 0
    assert_vis_equal(vis, oracle_vis(scene, cam), f"queue 1 of {capacity}")
    del keep


@pytest.mark.parametrize("s2", [32, 1023, 1024, 4096, 1 << 20])
@pytest.mark.parametrize("n", [1, 31, 700, 20000])
def test_stage2_sizes(api, n, s2):
    """Queues dealt out singly and in groups, ranges about the 1024 pixels of the
    shared pixel loop and about the stage-2 limit, tiles with and without a
    covered pixel."""
    scene = _slivers(n, 1100, 1060, seed=100 + n, shapes=[(1, 1), (32, 32), (1025, 1), (33, 32), (300, 200), (15, 70),
                                                          (900, 900) if n < 1000 else (64, 64)])
    cam = scene.cameras[0]
    r = api.Renderer(0)
    r.set_config(stage1_max_pixels=1, stage2_max_pixels=s2, stage1_exact_all=1)
    keep = upload(r, scene, with_colour=False)
    vis = r.render(cam.view, cam.proj, cam.W, cam.H)
    r.sync()
    assert_vis_equal(vis, oracle_vis(scene, cam), f"{n} triangles, stage-2 limit {s2}")
    del keep


@pytest.mark.parametrize("size", [(3840, 2160), (1921, 1081), (8000, 37)])
def test_room_large(api, size):
    """Clipped triangles as wide as the screen: edge functions far beyond 32 bits."""
    W, H = size
    scene = S.scene_room()
    cam = Camera(scene.cameras[0].view, S.perspective(80.0, W / H, 0.05, 100.0), W, H)
    r = api.Renderer(0)
    keep = upload(r, scene, with_colour=False)
    vis = r.render(cam.view, cam.proj, W, H)
    r.sync()
    assert_vis_equal(vis, oracle_vis(scene, cam), f"room {W} x {H}")
    del keep


@pytest.mark.parametrize("ray", [0, 1])
@pytest.mark.parametrize("n", [1, 2, 33, 151, 152, 304, 607, 608, 609, 1215, 1217])
def test_stage2_shares(api, n, ray):
    """Short queues of triangles cut by the near plane and the guard band, each
    shared by sixteen warps down to one; parts counted once."""
    rng = np.random.default_rng(n)
    pos = rng.uniform(-1, 1, (n, 3, 3)) * (2.0, 2.0, 1.0) + (0.0, 0.0, -0.6)
    pos[::3] *= (40.0, 40.0, 1.0)
    idx = np.arange(3 * n, dtype=np.int32).reshape(n, 3)
    scene = Scene([Mesh(pos=torch.tensor(pos.reshape(-1, 3).astype(np.float32)), idx=torch.from_numpy(idx))],
                  [Instance(0, np.eye(4, dtype=np.float32))],
                  [Camera(np.eye(4, dtype=np.float32), S.perspective(90.0, 1.0, 1e-2, 10.0), 140, 100)])
    cam = scene.cameras[0]
    r = api.Renderer(0)
    r.set_config(stage1_max_pixels=1, stage2_max_pixels=64, tile_log2=4, stage1_exact_all=1, stage3_raycast=ray,
                 collect_stats=1)
    keep = upload(r, scene, with_colour=False)
    vis = r.render(cam.view, cam.proj, cam.W, cam.H)
    parts = r.sync()["queued_stage3"]
    ref = orc.render_paper(orc.OracleScene(scene), cam, 1, 64) if ray else oracle_vis(scene, cam)
    assert_vis_equal(vis, ref, f"{n} clipped triangles")
    again = r.render(cam.view, cam.proj, cam.W, cam.H)
    assert r.sync()["queued_stage3"] == parts
    assert torch.equal(vis, again)
    del keep
