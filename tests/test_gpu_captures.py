"""Frames captured by the caller give back what they hold when their graph is
gone, and a context with captured frames alive renders whatever it rendered
without them: larger tables, bitmaps and queues among it."""
import gc
import time

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


def _capture(api, r, view, vis, status=None):
    """The captured frame, or None where it was refused (with `status`, if one is expected)."""
    g = torch.cuda.CUDAGraph()
    ok = True
    with torch.cuda.stream(torch.cuda.Stream()):
        g.capture_begin(capture_error_mode="relaxed")
        try:
            r.render(*view, vis=vis)
        except api.CurastError as e:
            ok = False
            assert status is None or e.status == status
        g.capture_end()
    return g if ok else None


def _replay(g):
    torch.cuda.synchronize()
    g.replay()
    torch.cuda.synchronize()


@pytest.mark.filterwarnings("ignore:The CUDA Graph is empty")
def test_slots_come_back(api, scene):
    """Three are alive at a time, a fourth is refused by name, and any number
    one after the other is taken (the runtime tells of a graph's end a moment
    after it)."""
    r = api.Renderer()
    keep = upload(r, scene, with_colour=False)
    want = r.render(*_view())
    r.sync()
    vis = torch.zeros_like(want)
    graphs = [_capture(api, r, _view(), vis) for _ in range(3)]
    assert all(graphs)
    assert _capture(api, r, _view(), vis, status=-11) is None
    for _ in range(8):
        graphs.pop(0).reset()
        gc.collect()
        deadline = time.time() + 10.0
        g = None
        while g is None and time.time() < deadline:
            g = _capture(api, r, _view(), vis, status=-11)
            if g is None:
                time.sleep(0.01)
        assert g is not None, "the slot of a destroyed graph did not come back"
        graphs.append(g)
        vis.zero_()
        _replay(g)
        assert_vis_equal(vis, u64(want), "captured frame")
    del keep


def test_a_context_grows_beside_captured_frames(api, scene):
    """More pairs than the tables held, a larger bitmap and other queues: direct
    frames are those of a context without captures, and the captured frame's
    replays still its own."""
    r, plain = api.Renderer(), api.Renderer()
    keep = [upload(x, scene, with_colour=False) for x in (r, plain)]
    want = r.render(*_view())
    r.sync()
    vis = torch.zeros_like(want)
    graph = _capture(api, r, _view(), vis)
    assert graph
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
