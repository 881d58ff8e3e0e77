"""The path kernels on both sides of every line that chooses between them:
tiles or lanes by path length, triangles and lanes, and the two tile sizes.

The reference is one path per lane throughout: the one-trace step of a context
with a memory budget, which takes no scratch for tiles.  The same paths in the
same order give the same image bit for bit, whatever renders it, and the
FP64-accumulated gradients agree to the FP32 rounding of each term (2^-24
each, summed in FP64: 1e-6 of the largest)."""
import numpy as np
import pytest

from paper_2503_12174_gb300 import dpcs, scenes
from gpu_util import need_cuda

pytestmark = pytest.mark.gpu


def _scene(mesh, H, W, spp, bounces):
    if mesh == "corner":
        sc = scenes.corner(res=48, tex=24, spp=spp, bounces=bounces, seed=5)
    elif mesh == "sphere":
        sc = scenes.sphere(subdiv=3, res=48, spp=spp, bounces=bounces, seed=5)
    else:
        sc = scenes.heightfield(spp=spp, cam=32, proj=(40, 56), tex=32, n_vert=mesh).replace(bounces=bounces)
    return sc.replace(Kc=scenes.intrinsics(W, H, 40.0), Hc=H, Wc=W)


# lanes = pixels x 16 at 16 spp
CASES = [
    ("corner", 124, 252, 16, 3), ("corner", 125, 250, 16, 3),      # 499,968 and 500,000: the tile sizes
    ("corner", 124, 252, 16, 2), ("corner", 125, 250, 16, 2),      # two bounces: tiles, lanes
    ("corner", 124, 1008, 16, 2), ("corner", 125, 1000, 16, 2),    # 1,999,872 and 2,000,000: lanes, tiles
    ("corner", 248, 252, 16, 3), ("corner", 250, 250, 16, 3),      # 999,936 and 1,000,000: the replay
    ("sphere", 250, 250, 16, 4), ("sphere", 31, 33, 5, 8),
    (72, 125, 250, 16, 3), (73, 125, 250, 16, 3),                  # 10,082 and 10,368 triangles
    (101, 124, 252, 16, 3), (101, 125, 250, 16, 3),                # 20,000: renders in lanes, records in tiles
    ("corner", 125, 250, 17, 2), ("corner", 250, 250, 11, 2), ("corner", 40, 50, 3, 4),  # rounds of samples not full
    (73, 41, 43, 16, 1), (28, 250, 250, 16, 3), (29, 250, 250, 16, 3),  # one bounce; 1,458 and 1,568: the replay
]


@pytest.mark.parametrize("mesh,H,W,spp,bounces", CASES)
def test_every_route_renders_the_lanes_image(mesh, H, W, spp, bounces):
    torch = need_cuda()
    sc = _scene(mesh, H, W, spp, bounces)
    out = {}
    for budget in (0, 1 << 30):
        c = dpcs.Context(0, hbm_budget_bytes=budget)
        c.set_grad_accum(dpcs.DPCS_ACCUM_F64)
        h = c.upload(sc.verts, sc.tris, sc.uv)
        alb, rough, Ip = (torch.from_numpy(np.ascontiguousarray(x)).cuda() for x in (sc.albedo, sc.rough, sc.Ip))
        args = (h, alb, rough, Ip, dpcs.view_of(sc), dpcs.make_params(sc.params), spp, bounces, sc.seed)
        Ic, Ec, dIc, tgt = (torch.zeros((H, W, 3), device="cuda") for _ in range(4))
        tgt.fill_(0.05)
        loss = torch.zeros(1, device="cuda")
        try:
            for how in ("step",) if budget else ("step", "render", "keep", "replay"):
                g = [torch.zeros_like(x) for x in (Ip, alb, rough)]
                kw = dict(dIp=g[0], dAlbedo=g[1], dRough=g[2])
                if how == "step":
                    c.render_loss_backward(*args, tgt, loss, Ic=Ic, Ec=Ec, **kw)
                else:
                    c.render(*args, Ic=Ic, Ec=Ec, keep=how == "keep")
                    c.l2_loss(Ic, tgt, dIc, loss)
                    if how != "render":
                        c.render_backward(*args, Ec, Ic, dIc, kept=how == "keep", **kw)
                c.sync()
                out["lanes" if budget else how] = [Ic.cpu().numpy()] + [x.cpu().numpy().astype(np.float64) for x in g]
        finally:
            c.close()
    ref = out.pop("lanes")
    assert np.abs(ref[0]).max() > 0
    for how, got in out.items():
        np.testing.assert_array_equal(got[0], ref[0], err_msg=how)
        if how != "render":
            for x, y in zip(got[1:], ref[1:]):
                np.testing.assert_allclose(x, y, rtol=1e-5, atol=1e-6 * np.abs(y).max(), err_msg=how)


@pytest.mark.parametrize("mesh,H,W,spp,bounces", [c for c in CASES if c[4] == 2] + [CASES[0], CASES[1], CASES[10], CASES[11]])
def test_principled_render_gives_the_lanes_image(mesh, H, W, spp, bounces):
    torch = need_cuda()
    sc = scenes.with_principled(_scene(mesh, H, W, spp, bounces), seed=8)
    out = []
    for budget in (0, 1 << 30):
        c = dpcs.Context(0, hbm_budget_bytes=budget)
        h = c.upload(sc.verts, sc.tris, sc.uv)
        mat = [torch.from_numpy(np.ascontiguousarray(x)).cuda() for x in (sc.albedo, sc.rough, sc.metallic, sc.normal, sc.Ip)]
        args = (h, *mat, dpcs.view_of(sc), dpcs.make_params(sc.params), spp, bounces, sc.seed)
        Ic, tgt = torch.zeros((H, W, 3), device="cuda"), torch.zeros((H, W, 3), device="cuda")
        try:
            if budget:
                c.render_loss_backward_principled(*args, tgt, torch.zeros(1, device="cuda"), Ic=Ic,
                                                  dIp=torch.zeros_like(mat[4]))
            else:
                c.render_principled(*args, Ic=Ic)
            c.sync()
            out.append(Ic.cpu().numpy())
        finally:
            c.close()
    np.testing.assert_array_equal(out[0], out[1])
