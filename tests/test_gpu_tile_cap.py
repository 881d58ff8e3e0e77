"""The visit cap in the block-tile kernels: every step down the tree counts,
whether it meets a leaf or not, as in the lanes kernels.  Only valid trees are
walked here; the cap is set below what their rays need."""
import numpy as np
import pytest

from paper_2503_12174_gb300 import dpcs, scenes
from gpu_util import need_cuda

pytestmark = pytest.mark.gpu


def _limited(c):
    """Has a traversal since the last call met the cap?"""
    try:
        c.sync()
    except dpcs.DPCSError as e:
        assert e.status == dpcs.DPCS_ERR_TRAVERSAL_LIMIT
        return True
    return False


@pytest.mark.parametrize("how", ["render", "keep", "step", "replay", "principled"])
def test_cap_counts_steps_that_reach_no_leaf(how):
    """Four small triangles in two pairs: a ray between the triangles of the
    first pair takes two steps (the root, the pair's node) and meets no
    leaf.  A cap of one has to be reported, a cap of two not."""
    torch = need_cuda()
    sc = scenes.plane(res=16, spp=2)
    tri = np.array([[-0.05, -0.02, 1.0], [0.05, -0.02, 1.1], [0.0, 0.02, 1.05]], np.float32)
    verts = np.concatenate([tri + np.float32([x, y, 0]) for x in (0.0, 3.0) for y in (-0.6, 0.6)])
    uv = np.zeros((12, 2), np.float32)
    c = dpcs.Context(0)
    h = c.upload(verts, np.arange(12, dtype=np.int32).reshape(4, 3), uv)
    alb, rough, Ip = (torch.from_numpy(np.ascontiguousarray(x)).cuda() for x in (sc.albedo, sc.rough, sc.Ip))
    view, prm = dpcs.view_of(sc), dpcs.make_params(sc.params)
    Ic, Ec, tgt, dIc = (torch.ones((sc.Hc, sc.Wc, 3), device="cuda") for _ in range(4))
    loss, dIp = torch.zeros(1, device="cuda"), torch.zeros_like(Ip)
    args = (h, alb, rough, Ip, view, prm, sc.spp, 2, sc.seed)
    try:
        for cap in (1, 2):
            c.set_visit_cap(cap)
            if how in ("render", "keep"):
                c.render(*args, Ic=Ic, Ec=Ec, keep=how == "keep")
            elif how == "step":
                c.render_loss_backward(*args, tgt, loss, Ic=Ic, Ec=Ec, dIp=dIp)
            elif how == "replay":
                c.render_backward(*args, Ec, tgt, dIc, dIp=dIp)
            else:
                c.render_principled(h, alb, rough, None, None, Ip, view, prm, sc.spp, 2, sc.seed, Ic=Ic)
            assert _limited(c) == (cap == 1)
    finally:
        c.close()


@pytest.mark.parametrize("cap", [1, 2, 5, 9, 14, 20, 30, 60])
def test_capped_image_is_that_of_the_lanes(cap):
    """A capped ray misses, so the image tells where each ray was cut: the
    tiles' image equals that of the one-trace step under a memory budget,
    which runs one path per lane."""
    torch = need_cuda()
    sc = scenes.corner(res=32, tex=24, spp=8, bounces=3, seed=5)
    out = []
    for budget in (0, 1 << 30):
        c = dpcs.Context(0, hbm_budget_bytes=budget)
        h = c.upload(sc.verts, sc.tris, sc.uv)
        alb, rough, Ip = (torch.from_numpy(np.ascontiguousarray(x)).cuda() for x in (sc.albedo, sc.rough, sc.Ip))
        Ic, tgt = torch.empty((sc.Hc, sc.Wc, 3), device="cuda"), torch.zeros((sc.Hc, sc.Wc, 3), device="cuda")
        args = (h, alb, rough, Ip, dpcs.view_of(sc), dpcs.make_params(sc.params), sc.spp, sc.bounces, sc.seed)
        try:
            c.set_visit_cap(cap)
            if budget:
                c.render_loss_backward(*args, tgt, torch.zeros(1, device="cuda"), Ic=Ic, dIp=torch.zeros_like(Ip))
            else:
                c.render(*args, Ic=Ic)
            out.append((_limited(c), Ic.cpu().numpy()))
        finally:
            c.close()
    assert out[0][0] == out[1][0]
    np.testing.assert_array_equal(out[0][1], out[1][1])
