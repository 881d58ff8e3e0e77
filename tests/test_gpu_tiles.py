"""The block-tile path kernels against the lanes kernels on the same paths.

The server's relighting kernel traces one path per lane throughout, so a
relit image is the lanes kernel's; dpcs_render picks tiles by size.  Both add
the same values in the same order, so images are equal bit for bit, at sizes
around the tiles' edges: fewer lanes than a tile, a last tile of a few lanes,
samples that do not fill a round, either tile size, the longest paths."""
import numpy as np
import pytest

from paper_2503_12174_gb300 import dpcs, scenes
from gpu_util import need_cuda

pytestmark = pytest.mark.gpu


def _scene(mesh, H, W, spp, bounces):
    if mesh == "corner":
        sc = scenes.corner(res=32, tex=24, spp=spp, bounces=bounces, seed=5)
    elif mesh == "sphere":
        sc = scenes.sphere(subdiv=2, spp=spp, bounces=bounces, seed=5)
    elif mesh == "field":  # 20,000 triangles: past the renders' limit, within the record kernels
        sc = scenes.heightfield(spp=spp, cam=32, proj=(40, 56), tex=32, n_vert=101).replace(bounces=bounces)
    else:  # a single triangle: the tree has no inner node
        sc = scenes.plane(res=32, spp=spp, seed=5)
        sc = sc.replace(tris=sc.tris[:1], bounces=bounces)
    return sc.replace(Kc=scenes.intrinsics(W, H, 40.0), Hc=H, Wc=W)


@pytest.mark.parametrize("mesh,H,W,spp,bounces", [
    ("corner", 1, 1, 1, 2), ("corner", 1, 3, 7, 3), ("corner", 5, 13, 1, 8), ("corner", 17, 31, 35, 3),
    ("corner", 9, 57, 64, 2), ("corner", 127, 123, 32, 3), ("corner", 125, 125, 33, 3), ("corner", 128, 123, 33, 4),
    ("sphere", 24, 24, 16, 8), ("triangle", 20, 20, 8, 3)])
def test_tiles_render_what_lanes_render(mesh, H, W, spp, bounces):
    torch = need_cuda()
    sc = _scene(mesh, H, W, spp, bounces)
    c = dpcs.Context(0)
    h = c.upload(sc.verts, sc.tris, sc.uv)
    alb, rough, Ip = (torch.from_numpy(np.ascontiguousarray(x)).cuda() for x in (sc.albedo, sc.rough, sc.Ip))
    view, prm = dpcs.view_of(sc), dpcs.make_params(sc.params)
    srv = dpcs.Server(c)
    try:
        Ic, _ = c.render(h, alb, rough, Ip, view, prm, spp, bounces, sc.seed)
        c.sync()
        out = torch.empty((H, W, 3)).pin_memory()
        slot = srv.add_scene(h, alb, rough, view, prm, bounces)
        srv.submit(dpcs.DPCS_REQ_RELIGHT, slot, H, W, spp, sc.seed, torch.from_numpy(sc.Ip), out)
        srv.drain()
        assert torch.equal(Ic.cpu(), out) and (mesh == "triangle" or H * W < 100 or out.abs().max() > 0)
    finally:
        srv.close()
        c.free(h)
        c.close()


@pytest.mark.parametrize("mesh,H,W,spp,bounces", [
    ("corner", 1, 1, 1, 2), ("corner", 1, 3, 7, 3), ("corner", 17, 31, 35, 3), ("corner", 9, 57, 100, 3),
    ("corner", 125, 125, 33, 3), ("corner", 12, 11, 300, 3), ("sphere", 24, 24, 16, 8), ("triangle", 20, 20, 8, 3),
    ("field", 31, 29, 8, 4)])
def test_tile_gradients_equal_lane_gradients(mesh, H, W, spp, bounces):
    """A context with a memory budget gets no scratch for the tiles' records
    and runs the lanes kernels: the same paths, so the image is equal bit for
    bit and the FP64-accumulated gradients to FP32 rounding of each term
    (2^-24 each, summed in FP64: 1e-6 of the largest), for the one-trace step
    and for the separate calls, with one round and several, below and above
    the one-trace step's record limit (300 spp)."""
    torch = need_cuda()
    sc = _scene(mesh, H, W, spp, bounces)
    out = []
    for budget in (0, 1 << 30):
        c = dpcs.Context(0, hbm_budget_bytes=budget)
        c.set_grad_accum(dpcs.DPCS_ACCUM_F64)
        h = c.upload(sc.verts, sc.tris, sc.uv)
        alb, rough, Ip = (torch.from_numpy(np.ascontiguousarray(x)).cuda() for x in (sc.albedo, sc.rough, sc.Ip))
        view, prm = dpcs.view_of(sc), dpcs.make_params(sc.params)
        tgt = torch.full((H, W, 3), 0.05, device="cuda")
        Ec, Ic, dIc, loss = torch.empty_like(tgt), torch.empty_like(tgt), torch.empty_like(tgt), torch.zeros(1, device="cuda")
        try:
            for fused in (True, False):
                g = [torch.zeros_like(Ip), torch.zeros_like(alb), torch.zeros_like(rough), torch.zeros(11, device="cuda")]
                kw = dict(dIp=g[0], dAlbedo=g[1], dRough=g[2], dParams=g[3])
                if fused:
                    c.render_loss_backward(h, alb, rough, Ip, view, prm, spp, bounces, sc.seed, tgt, loss, Ic=Ic, Ec=Ec, **kw)
                else:
                    c.render(h, alb, rough, Ip, view, prm, spp, bounces, sc.seed, Ic=Ic, Ec=Ec)
                    c.l2_loss(Ic, tgt, dIc, loss)
                    c.render_backward(h, alb, rough, Ip, view, prm, spp, bounces, sc.seed, Ec, Ic, dIc, **kw)
                c.sync()
                out.append([Ic.cpu().numpy().copy(), loss.item()] + [x.cpu().numpy().astype(np.float64) for x in g])
            c.free(h)
        finally:
            c.close()
    for a, b in ((out[0], out[2]), (out[1], out[3]), (out[0], out[1])):
        np.testing.assert_array_equal(a[0], b[0])
        assert abs(a[1] - b[1]) <= 1e-6 * abs(b[1])
        for x, y in zip(a[2:], b[2:]):
            np.testing.assert_allclose(x, y, rtol=1e-5, atol=1e-6 * np.abs(y).max())


@pytest.mark.parametrize("mesh,H,W,spp,bounces,maps", [
    ("corner", 1, 3, 7, 3, "both"), ("corner", 17, 31, 35, 3, "both"), ("corner", 9, 57, 100, 2, "metallic"),
    ("corner", 125, 125, 33, 3, "both"), ("corner", 12, 11, 300, 3, "normal"), ("sphere", 24, 24, 16, 8, "both"),
    ("triangle", 20, 20, 8, 3, "both"), ("field", 31, 29, 8, 4, "both")])
def test_principled_tiles_equal_lanes(mesh, H, W, spp, bounces, maps):
    """As above with the principled material, whose render and kept records
    run in tiles with or without a budget: one-trace step, separate calls and
    kept records against a budget's one-trace and separate steps.  Images are
    equal bit for bit.  The FP32 gradient accumulators add n terms in any
    order, so they differ by at most n 2^-23 of the terms' absolute sum, n
    their number per texel; four times the largest gradient stands for that sum."""
    torch = need_cuda()
    sc = scenes.with_principled(_scene(mesh, H, W, spp, bounces), seed=8)
    out = []
    for budget in (0, 1 << 30):
        c = dpcs.Context(0, hbm_budget_bytes=budget)
        h = c.upload(sc.verts, sc.tris, sc.uv)
        alb, rough, Ip, met, nrm = (torch.from_numpy(np.ascontiguousarray(x)).cuda()
                                    for x in (sc.albedo, sc.rough, sc.Ip, sc.metallic, sc.normal))
        met, nrm = (None if maps == "normal" else met), (None if maps == "metallic" else nrm)
        view, prm = dpcs.view_of(sc), dpcs.make_params(sc.params)
        tgt = torch.full((H, W, 3), 0.05, device="cuda")
        Ec, Ic, dIc, loss = torch.empty_like(tgt), torch.empty_like(tgt), torch.empty_like(tgt), torch.zeros(1, device="cuda")
        args = (h, alb, rough, met, nrm, Ip, view, prm, spp, bounces, sc.seed)
        try:
            for how in ("one", "two", "kept"):
                g = [torch.zeros_like(x) for x in (Ip, alb, rough, alb[..., 0], alb)]
                kw = dict(dIp=g[0], dAlbedo=g[1], dRough=g[2], dMetallic=None if met is None else g[3],
                          dNormal=None if nrm is None else g[4])
                if how == "one":
                    c.render_loss_backward_principled(*args, tgt, loss, Ic=Ic, Ec=Ec, **kw)
                else:
                    c.render_principled(*args, Ic=Ic, Ec=Ec, keep=how == "kept")
                    c.l2_loss(Ic, tgt, dIc, loss)
                    c.render_backward_principled(*args, Ec, Ic, dIc, kept=how == "kept", **kw)
                c.sync()
                out.append([Ic.cpu().numpy().copy(), Ec.cpu().numpy().copy()] + [x.cpu().numpy().astype(np.float64) for x in g])
            c.free(h)
        finally:
            c.close()
    n = 4.0 * H * W * spp * bounces / min(sc.rough.size, sc.Ip.size // 3) + 4
    ref = out[3]
    for a in out:
        np.testing.assert_array_equal(a[0], ref[0])
        np.testing.assert_array_equal(a[1], ref[1])
        for x, y in zip(a[2:], ref[2:]):
            np.testing.assert_allclose(x, y, rtol=1e-5, atol=4 * n * 2.0 ** -23 * np.abs(y).max())
