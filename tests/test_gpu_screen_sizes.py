"""The screen passes at the image sizes where their split changes (one, two and
four rows a thread), at odd sizes, over several instances, and the backward's
grouping from one triangle a pixel to one triangle over many."""
import numpy as np
import pytest
import torch

import synthetic as S
from oracle import adjoint as A
from oracle import oracle as orc
from synthetic.scenes import Camera, Instance, Scene

from gpu_util import u64, upload

pytestmark = pytest.mark.gpu

SIZES = [(1, 1), (33, 7), (299, 201), (641, 479), (2003, 2001)]


@pytest.fixture(scope="module")
def api():
    import __graft_entry__ as g
    g.build()
    from paper_2604_21749_gb300 import api as A_
    return A_


def _scene(W, H):
    hf, sp = S.heightfield_mesh(60, seed=4), S.sphere_mesh(20, seed=5)
    inst = []
    for k in range(5):
        m = np.eye(4, dtype=np.float32)
        m[:3, 3] = (0.9 * (k % 3) - 0.9, 0.05 * k, 0.8 * (k // 3))
        if k % 2:
            m[:3, :3] *= 0.2
        inst.append(Instance(k % 2, m))
    cam = Camera(S.look_at((0.5, 1.6, -1.4), (0.4, 0.0, 0.6)), S.perspective(70.0, W / H, 0.01, 100.0), W, H)
    return Scene([hf, sp], inst, [cam])


@pytest.mark.parametrize("size", SIZES)
def test_resolves(api, size):
    W, H = size
    sc = _scene(W, H)
    cam = sc.cameras[0]
    r = api.Renderer(0)
    keep = upload(r, sc)
    osc = orc.OracleScene(sc)
    vis = r.render(cam.view, cam.proj, W, H)
    ref = orc.render(osc, cam)
    f32, u8 = r.resolve(cam.view, cam.proj, vis)
    rf, r8 = orc.resolve(osc, cam, ref)
    np.testing.assert_array_equal(u8.cpu().numpy(), r8)
    np.testing.assert_allclose(f32.cpu().numpy(), rf, atol=1e-6, rtol=0)
    tex = [(S.grid_uv(60), S.texture_mip_chain(7, seed=1), 7), None]
    uv, tx = tex[0][0].cuda(), tex[0][1].cuda()
    r.set_mesh_texture(0, uv, tx, 7)
    f32, u8, lev = r.resolve_textured(cam.view, cam.proj, vis)
    rf, r8, rl = orc.resolve_textured(osc, cam, ref, tex)
    np.testing.assert_array_equal(lev.cpu().numpy(), rl)
    np.testing.assert_array_equal(u8.cpu().numpy(), r8)
    np.testing.assert_allclose(f32.cpu().numpy(), rf, atol=1e-6, rtol=0)
    del keep


@pytest.mark.parametrize("ss", [1, 2, 3, 5, 7, 8])
@pytest.mark.parametrize("size", [(1, 1), (33, 7), (131, 77)])
def test_supersampled(api, size, ss):
    W, H = size
    sc = _scene(W, H)
    cam = sc.cameras[0]
    fine = Camera(cam.view, cam.proj, ss * W, ss * H)
    r = api.Renderer(0)
    keep = upload(r, sc)
    osc = orc.OracleScene(sc)
    vis = r.render(fine.view, fine.proj, fine.W, fine.H)
    f32, u8 = r.resolve_ss(cam.view, cam.proj, vis, ss)
    rf, r8 = orc.resolve_ss(osc, fine, orc.render(osc, fine), ss)
    np.testing.assert_array_equal(u8.cpu().numpy(), r8)
    np.testing.assert_allclose(f32.cpu().numpy(), rf, atol=1e-6, rtol=0)
    del keep


@pytest.mark.parametrize("want", ["both", "attr", "pos"])
@pytest.mark.parametrize("C", [1, 3, 4, 5, 16])
@pytest.mark.parametrize("n,size", [(2, (157, 93)), (40, (157, 93)), (300, (157, 93)), (40, (701, 450)), (1, (1, 1))])
def test_interpolation(api, n, size, C, want):
    W, H = size
    hf = S.heightfield_mesh(n, seed=31)
    cam = Camera(S.look_at((0.5, 1.1, -0.25), (0.5, 0.0, 0.55)), S.perspective(55.0, W / H, 1e-2, 100.0), W, H)
    sc = Scene([S.sphere_mesh(6, seed=2), hf], [Instance(0, np.diag([0.05, 0.05, 0.05, 1.0]).astype(np.float32)),
                                               Instance(1, np.eye(4, dtype=np.float32))], [cam])
    rng = np.random.default_rng(C)
    attr = rng.uniform(-1, 1, size=(hf.V, C)).astype(np.float32)
    r = api.Renderer(0)
    keep = upload(r, sc, with_colour=False)
    vis = r.render(cam.view, cam.proj, W, H)
    osc = orc.OracleScene(sc)
    out = r.interpolate(1, cam.view, cam.proj, vis, torch.from_numpy(attr).cuda())
    wf, _ = orc.interpolate(osc, cam, orc.render(osc, cam), 1, attr)
    np.testing.assert_allclose(out.cpu().numpy(), wf, atol=1e-6 * 8, rtol=0)   # attributes up to 1, extrapolated up to 8 times
    g = rng.normal(size=(H, W, C)).astype(np.float32)
    ga, gp = r.interpolate_backward(1, cam.view, cam.proj, vis, torch.from_numpy(attr).cuda(), torch.from_numpy(g).cuda(),
                                    want_attr=want != "pos", want_pos=want != "attr")
    assert (ga is None) == (want == "pos") and (gp is None) == (want == "attr")
    fx, fy, _ = orc.camera_params(cam.proj)
    mv = orc.model_view(cam.view, np.eye(4, dtype=np.float32))
    tri = A.pixel_triangles(u64(vis), sc.meshes[0].T, hf.T)
    da, dp = A.adjoint64(hf.pos.numpy(), hf.idx.numpy(), attr, mv, fx, fy, W, H, tri, g.astype(np.float64).reshape(-1, C))
    for got, ref in ((ga, da), (gp, dp)):
        if got is not None:
            assert np.linalg.norm(got.cpu().numpy() - ref) <= 1e-4 * max(np.linalg.norm(ref), 1e-30)
    del keep


@pytest.mark.parametrize("n", [1, 7, 16])
def test_instances_as_parameters(api, n):
    """Up to sixteen instances travel as kernel parameters; the same ones
    followed by others that are out of sight go up as tables: same images."""
    W, H = 333, 210
    hf, sp = S.heightfield_mesh(40, seed=4), S.sphere_mesh(16, seed=5)
    inst = []
    for k in range(17):
        m = np.eye(4, dtype=np.float32)
        m[:3, 3] = (0.7 * (k % 3) - 0.7, 0.05 * k, 0.6 * (k // 3)) if k < n else (0.0, 0.0, -500.0 - 9 * k)
        inst.append(Instance(k % 2, m))
    cam = Camera(S.look_at((0.5, 1.6, -1.4), (0.4, 0.0, 0.6)), S.perspective(70.0, W / H, 0.01, 100.0), W, H)
    uv, tx = S.grid_uv(40).cuda(), S.texture_mip_chain(6, seed=1).cuda()
    attr = torch.rand((hf.pos.shape[0], 3), generator=torch.Generator().manual_seed(1)).cuda()
    got = []
    for count in (n, 17):
        r = api.Renderer(0)
        keep = upload(r, Scene([hf, sp], inst[:count], [cam]), compressed=(1,))
        vis = r.render(cam.view, cam.proj, W, H)
        out = [vis, *r.resolve(cam.view, cam.proj, vis)]
        out.append(r.interpolate(0, cam.view, cam.proj, vis, attr))
        out += r.resolve_ss(cam.view, cam.proj, vis, 3) if W % 3 == 0 and H % 3 == 0 else []
        r.set_mesh_texture(0, uv, tx, 6)
        out += r.resolve_textured(cam.view, cam.proj, vis)
        ga, gp = r.interpolate_backward(0, cam.view, cam.proj, vis, attr, torch.ones((H, W, 3), device="cuda"))
        got.append((out, ga))
        r.sync()
        del keep
    assert (got[0][0][0] != -1).any() and got[0][0][3].abs().sum() > 0
    for a, b in zip(got[0][0], got[1][0]):
        assert torch.equal(a, b)
    # sums of at most W H terms, nearly all of one sign, in any order
    torch.testing.assert_close(got[0][1], got[1][1], rtol=2 * W * H * 2.0 ** -24, atol=1e-4)
