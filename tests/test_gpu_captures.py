"""A context with captured frames alive renders whatever it rendered without
them: larger tables, bitmaps and queues among it."""
import numpy as np
import pytest
import torch

import synthetic as S

from gpu_util import assert_vis_equal, u64, upload

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def api():
    import __graft_entry__ as g
    g.build()
    from paper_2604_21749_gb300 import api as A
    return A


@pytest.fixture(scope="module")
def scene():
    return S.scene_batched(n_meshes=4, n_instances=24, tmin=500, tmax=4e3, views=((160, 90),), seed=5)


def _view(k=0):
    return (S.look_at((60.0 * (k % 3 - 1), 6.0 + 3 * k, -70.0 + 9 * k), (0, 0, 0)), S.perspective(60, 1.6, 0.1, 500.0),
            97 + 16 * k, 61 + 8 * k)


def _capture(r, view, vis):
    g = torch.cuda.CUDAGraph()
    with torch.cuda.stream(torch.cuda.Stream()):
        g.capture_begin(capture_error_mode="relaxed")
        r.render(*view, vis=vis)
        g.capture_end()
    return g


def _replay(g):
    torch.cuda.synchronize()
    g.replay()
    torch.cuda.synchronize()


def test_a_context_grows_beside_captured_frames(api, scene):
    """More pairs than the tables held, a larger bitmap and other queues: direct
    frames are those of a context without captures, and the captured frame's
    replays still its own."""
    r, plain = api.Renderer(), api.Renderer()
    keep = [upload(x, scene, with_colour=False) for x in (r, plain)]
    want = r.render(*_view())
    r.sync()
    vis = torch.zeros_like(want)
    graph = _capture(r, _view(), vis)
    rng = np.random.default_rng(2)
    for step in range(3):
        for _ in range(400):
            m = np.eye(4, dtype=np.float32)
            m[:3, 3] = rng.uniform(-30, 30, size=3)
            for x in (r, plain):
                x.add_instance(step % 4, m)
        if step == 2:
            r.set_config(queue1_capacity=1 << 16, queue2_capacity=1 << 16, stage3_tile_buffer=1)
        v = _view(step)
        assert_vis_equal(r.render(*v), u64(plain.render(*v)), "direct frame beside a captured one")
        vis.zero_()
        _replay(graph)
        assert_vis_equal(vis, u64(want), f"replay after growth {step}")
    del keep
