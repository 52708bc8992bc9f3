"""Frames issued ahead of the device, frames of many views, frames without
triangles and frames captured by the caller: the words of each equal those of
the same frame rendered alone (bit-exact)."""
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


def _views(n):
    return [(S.look_at((60.0 * (k % 3 - 1), 6.0 + 3 * k, -70.0 + 9 * k), (0, 0, 0)),
             S.perspective(60, 1.6, 0.1, 500.0), 97 + 16 * k, 61 + 8 * k) for k in range(n)]


def _alone(r, views):
    out = []
    for v in views:
        out.append(r.render(*v))
        r.sync()
    return out


def test_frames_issued_ahead(api, scene):
    """More frames in a row than there are table copies, none waited for."""
    r = api.Renderer()
    keep = upload(r, scene, with_colour=False)
    views = _views(11)
    want = _alone(r, views)
    got = [r.render(*v) for v in views]
    r.sync()
    for k, (a, b) in enumerate(zip(got, want)):
        assert_vis_equal(a, u64(b), f"frame {k}")
    assert any((w != -1).any() for w in want)
    del keep


@pytest.mark.parametrize("n,graph", [(8, False), (9, False), (9, True)])
def test_many_views_are_cleared(api, scene, n, graph):
    """As many views as one launch clears, and one more; dirty buffers."""
    r = api.Renderer()
    keep = upload(r, scene, with_colour=False)
    views = _views(n)
    want = _alone(r, views)
    bufs = [torch.zeros_like(w) for w in want]
    for _ in range(2):
        out = r.render_batch([v + (b,) for v, b in zip(views, bufs)], use_graph=graph)
    r.sync()
    for k, (a, b) in enumerate(zip(out, want)):
        assert_vis_equal(a, u64(b), f"view {k}")
    del keep


def test_stage_times_of_an_empty_frame(api, scene):
    r = api.Renderer()
    v = _views(1)[0]
    r.render(*v)
    assert all(t >= 0.0 for t in r.stage_times()) and sum(r.stage_times()) < 100.0
    keep = upload(r, scene, with_colour=False)
    r.render(*v)
    t = r.stage_times()
    assert all(x >= 0.0 for x in t) and 0.0 < sum(t) < 1000.0
    del keep


def test_captured_frames(api, scene):
    """A frame captured by the caller replays its own camera after others were
    rendered; a fourth one is refused; direct frames go on."""
    r = api.Renderer()
    keep = upload(r, scene, with_colour=False)
    views = _views(8)
    want = _alone(r, views)
    s = torch.cuda.Stream()
    graphs, bufs = [], [torch.zeros_like(w) for w in want[:4]]
    torch.cuda.synchronize()
    with torch.cuda.stream(s):
        for k in range(4):
            g = torch.cuda.CUDAGraph()
            g.capture_begin(capture_error_mode="relaxed")
            refused = False
            try:
                r.render(*views[k], vis=bufs[k])
            except api.CurastError:
                refused = True
            g.capture_end()
            assert refused == (k == 3)
            graphs.append(g)
    for v, w in zip(views, want):
        assert_vis_equal(r.render(*v), u64(w), "direct frame after a capture")
    torch.cuda.synchronize()
    with torch.cuda.stream(s):
        for g in (graphs[1], graphs[0], graphs[2]):
            g.replay()
    torch.cuda.synchronize()
    for k in range(3):
        assert_vis_equal(bufs[k], u64(want[k]), f"captured frame {k}")
    del keep
