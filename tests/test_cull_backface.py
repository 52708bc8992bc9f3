"""The back-face rule of the instanced cull against the oracle's exact snapping
(CPU), and the cull's strip orders against the oracle's buffers (GPU).

The rule drops a triangle whose estimated doubled area lies below
-(4.01 m (dX + dY) + 8.01 m^2 + 2^-20 dX dY), m the margin and dX, dY the
estimated extents.  It is sound if the exact snapped area is then negative:
the restatement of the estimate in test_cull_bounds is sampled over triangles
of all sizes about the size of the margin and up."""
import numpy as np
import pytest
import torch

import synthetic as S
from oracle import oracle as orc
from synthetic.scenes import Camera, Instance, Mesh, Scene
from test_cull_bounds import F32, SETUPS, _constants, _exact, _f32, _fma, _rcp, _row


def _dropped(setup, scale, n=40000):
    """(triangles the rule drops, of these the ones whose exact area is not negative)."""
    cam, model, lo, hi, _ = setup
    cp = orc.camera_params(np.asarray(cam.proj, np.float32))
    mv = orc.model_view(np.asarray(cam.view, np.float32), model)
    rows, k, ws, win, _ = _constants(mv, lo, hi, cp, cam.W, cam.H)
    rng = np.random.default_rng(23)
    size = 10.0 ** rng.uniform(-6, -1, size=(n, 1, 1)) * (hi - lo)
    pts = np.clip(rng.uniform(lo, hi, size=(n, 1, 3)) + rng.uniform(-1, 1, size=(n, 3, 3)) * size, lo, hi).astype(F32)
    Xe, Ye, inside = _exact(mv, cp, cam, pts)
    area = (Xe[:, 1] - Xe[:, 0]) * (Ye[:, 2] - Ye[:, 0]) - (Xe[:, 2] - Xe[:, 0]) * (Ye[:, 1] - Ye[:, 0])
    x, y, z = pts[..., 0], pts[..., 1], pts[..., 2]
    xw, yw, w = _row(rows[0], x, y, z), _row(rows[1], x, y, z), _row(rows[2], x, y, z)
    dropped = wrong = 0
    for s in (-1, 1):
        r = _rcp(w, s)
        X, Y = _f32(xw * r), _f32(yw * r)
        a = np.maximum(np.abs(X).max(1), np.abs(Y).max(1))
        m = _f32(_fma(r.max(1), _fma(k[1], a, k[0]), _fma(k[2], a, k[3])).astype(np.float64) * scale)
        dX, dY = _f32(X.max(1) - X.min(1)), _f32(Y.max(1) - Y.min(1))
        ux, uy, vx, vy = X[:, 1] - X[:, 0], Y[:, 1] - Y[:, 0], X[:, 2] - X[:, 0], Y[:, 2] - Y[:, 0]
        est = _f32(_f32(ux * vy) - _f32(uy * vx))
        t = _fma(m, _fma(F32(8.01), m, _f32(F32(4.01) * _f32(dX + dY))), _f32(_f32(F32(2.0 ** -20) * dX) * dY))
        hit = (w.min(1) > ws) & (a < win) & (est < -t)
        assert inside[hit].all()
        dropped += int(hit.sum())
        wrong += int((area[hit] >= 0).sum())
    return dropped, wrong


@pytest.mark.parametrize("setup", SETUPS, ids=[s[-1] for s in SETUPS])
def test_dropped_triangles_face_away_exactly(setup):
    dropped, wrong = _dropped(setup, 1.0)
    assert dropped > 0
    assert wrong == 0, f"{wrong} of {dropped} dropped triangles do not face away in the exact path"


def test_a_margin_far_too_small_is_caught():
    """The sample is sharp enough to see a rule that forgets the margin."""
    assert sum(_dropped(s, 0.01, 20000)[1] for s in SETUPS) > 0


def _order(idx, order):
    """The cells' triangles in the listed order: as generated, facing the
    other way round, along the other diagonal, or the triangles shuffled."""
    if order == "rows":
        return idx
    if order == "flipped":
        return idx[:, [0, 2, 1]].contiguous()
    v00, v01, v10, v11 = idx[0::2, 0], idx[0::2, 1], idx[0::2, 2], idx[1::2, 2]
    if order == "diagonal":
        return torch.stack([v00, v01, v11, v00, v11, v10], dim=1).reshape(-1, 3).contiguous()
    if order == "mixed":                              # a row of each
        out = idx.clone()
        out[100:300] = _order(idx, "diagonal")[100:300]
        out[400:] = _order(idx, "flipped")[400:]
        return out
    return idx[torch.from_numpy(np.random.default_rng(3).permutation(idx.shape[0]))].contiguous()


@pytest.mark.gpu
@pytest.mark.parametrize("compressed", [False, True])
@pytest.mark.parametrize("copies", [1, 2, 70])
@pytest.mark.parametrize("order", ["rows", "flipped", "diagonal", "mixed", "shuffled"])
def test_strip_orders(order, copies, compressed):
    """Every strip order, single and instanced (group test on and off), partial
    groups at the mesh's end, seen from above and from below."""
    import __graft_entry__ as g
    g.build()
    from gpu_util import assert_vis_equal, decoded_scene, oracle_vis, upload
    from paper_2604_21749_gb300 import api
    hf = S.heightfield_mesh(37, seed=9)
    mesh = Mesh(pos=hf.pos, idx=_order(hf.idx, order))
    rng = np.random.default_rng(copies)
    inst = []
    for k in range(copies):
        m = np.eye(4)
        m[:3, :3] = S.scenes._random_rotation(rng) * rng.uniform(0.2, 1.5) if k else np.eye(3)
        m[:3, 3] = rng.uniform(-2, 2, size=3) if k else 0
        inst.append(Instance(0, m.astype(np.float32)))
    W, H = 333, 201
    cams = [Camera(S.look_at((0.5, y, -1.2), (0.5, 0.0, 0.5)), S.perspective(60.0, W / H, 0.01, 100.0), W, H)
            for y in (1.5, -1.5)]
    scene = Scene([mesh], inst, cams)
    comp = (0,) if compressed else ()
    ref = decoded_scene(scene, comp) if compressed else scene
    for group in (2, 0):
        r = api.Renderer(0)
        r.set_config(stage1_group_min_pairs=group)
        keep = upload(r, scene, with_colour=False, compressed=comp)
        for cam in cams:
            vis = r.render(cam.view, cam.proj, W, H)
            r.sync()
            assert_vis_equal(vis, oracle_vis(ref, cam), f"{order}, {copies} copies")
        del keep
