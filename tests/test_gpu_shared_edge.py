"""Rays exactly through an edge that two triangles share.

Such a ray may hit both triangles at the same t; the triangle of the lower
index wins, and the hit's barycentrics have to be that triangle's.  The scene
is a pair (or a field of pairs) of coplanar triangles whose shared edge lies in
the plane x = y, seen through pixel centres, so that every ray of the image's
diagonal has x = y to the last bit.  Which triangle wins does not change the
surface point, its texel or its normal, so the image is the oracle's; one
triangle's barycentrics in the other would put the point somewhere else on it."""
import numpy as np
import pytest

from paper_2503_12174_gb300 import dpcs, scenes
from gpu_util import need_cuda

pytestmark = pytest.mark.gpu

RES = 64


def edge_scene(seed, swap):
    """Two triangles (A, B, C) and (A, C, D) in a tilted plane, A and C on
    x = y past the image's corners; swap: listed the other way round."""
    rng = np.random.default_rng(seed)
    p, q, z0 = rng.uniform(-0.4, 0.4), rng.uniform(-0.4, 0.4), rng.uniform(0.9, 1.6)
    r = rng.uniform(0.6, 1.1, 4) * z0
    xy = np.array([[-r[0], -r[0]], [r[1], -r[1] * rng.uniform(0.7, 1.2)], [r[2], r[2]],
                   [-r[3], r[3] * rng.uniform(0.7, 1.2)]])
    verts = np.concatenate([xy, (z0 + p * xy[:, :1] + q * xy[:, 1:])], 1).astype(np.float32)
    uv = (0.5 + 0.3 * xy / z0).astype(np.float32)  # affine in x and y: the same over both triangles
    tris = np.array([[0, 1, 2], [0, 2, 3]], np.int32)
    sc = scenes.plane(res=RES, spp=1)
    g = (np.arange(48) + 0.5) / 48
    alb = np.stack([0.2 + 0.7 * np.broadcast_to(g, (48, 48)), 0.9 - 0.7 * np.broadcast_to(g[:, None], (48, 48)),
                    0.3 + 0.5 * g[:, None] * g], -1).astype(np.float32)
    return sc.replace(verts=verts, uv=uv, tris=tris[::-1].copy() if swap else tris, albedo=alb,
                      rough=np.full((48, 48), 0.5, np.float32), Ip=np.full((RES, RES, 3), 0.8, np.float32),
                      params=scenes.Params(gamma_p=(2.2,) * 3, k_proj=4.0, ks=0.0, jitter=0), bounces=2)


def diagonal_image(sc, how, bounces):
    """Ec of the diagonal's pixels: c.render, or the one-trace step under a
    memory budget (one path per lane), of either material."""
    import torch

    c = dpcs.Context(0, hbm_budget_bytes=0 if how in ("render", "keep", "principled", "wavefront") else 1 << 30)
    try:
        if how == "wavefront":
            c.set_render_path(dpcs.DPCS_PATH_WAVEFRONT)
        h = c.upload(sc.verts, sc.tris, sc.uv)
        alb, rough, Ip = (torch.from_numpy(np.ascontiguousarray(x)).cuda() for x in (sc.albedo, sc.rough, sc.Ip))
        view, prm = dpcs.view_of(sc), dpcs.make_params(sc.params)
        Ic, Ec, tgt = (torch.zeros((sc.Hc, sc.Wc, 3), device="cuda") for _ in range(3))
        loss, dIp = torch.zeros(1, device="cuda"), torch.zeros_like(Ip)
        tail = (Ip, view, prm, 1, bounces, sc.seed)
        if how in ("render", "wavefront", "keep"):
            c.render(h, alb, rough, *tail, Ic=Ic, Ec=Ec, keep=how == "keep")
        elif how == "principled":
            c.render_principled(h, alb, rough, None, None, *tail, Ic=Ic, Ec=Ec)
        elif how == "step":
            c.render_loss_backward(h, alb, rough, *tail, tgt, loss, Ic=Ic, Ec=Ec, dIp=dIp)
        else:
            c.render_loss_backward_principled(h, alb, rough, None, None, *tail, tgt, loss, Ic=Ic, Ec=Ec, dIp=dIp)
        c.sync()
        return Ec.cpu().numpy()[np.arange(sc.Hc), np.arange(sc.Hc)].astype(np.float64)
    finally:
        c.close()


@pytest.mark.parametrize("how,bounces", [("render", 2), ("keep", 2), ("principled", 2), ("render", 1), ("principled", 1),
                                         ("keep", 1), ("step", 2), ("step principled", 2), ("wavefront", 2)])
def test_shared_edge_hits_keep_their_barycentrics(orc, how, bounces):
    """Within the tolerance of the image parity tests (1e-4 of the value) on
    every pixel of the diagonal, in both listings of the pair."""
    need_cuda()
    for seed in range(24):
        for swap in (False, True):
            sc = edge_scene(seed, swap)
            ref, _ = orc.render(sc, pixels=np.arange(RES) * (RES + 1), bounces=bounces)
            got = diagonal_image(sc, how, bounces)
            assert (ref.max(-1) > 0).sum() > RES // 2
            np.testing.assert_allclose(got, ref, rtol=1e-4, atol=1e-6, err_msg=f"seed {seed} swap {swap}")
