"""One iteration of the server with requests of every kind of launch: relights
that run in tiles because together they fill the chip, the same ones when they
do not, and those that always run in lanes (one bounce, a large tree).  Each
image equals, bit for bit, the request's own one-trace step in a context with
a memory budget, which runs one path per lane."""
import numpy as np
import pytest

from paper_2503_12174_gb300 import dpcs, scenes
from gpu_util import need_cuda

pytestmark = pytest.mark.gpu


def _resident(torch, c):
    """(scene, handle, maps) of a corner with three bounces and with two, a
    20,000-triangle field, and a plane with one bounce"""
    out = []
    field = scenes.heightfield(spp=1, cam=32, proj=(40, 56), tex=32, n_vert=101)
    corner = scenes.corner(res=32, tex=24)
    for sc, b in ((corner, 3), (corner, 2), (field, 4), (scenes.plane(res=32), 1)):
        maps = [torch.from_numpy(np.ascontiguousarray(x)).cuda() for x in (sc.albedo, sc.rough)]
        out.append((sc.replace(bounces=b), c.upload(sc.verts, sc.tris, sc.uv), maps))
    return out


@pytest.mark.parametrize("sizes", [
    [(0, 128, 32), (0, 33, 5), (1, 100, 16), (2, 57, 9), (3, 64, 4)],  # 688,644 lanes may run in tiles
    [(0, 120, 32), (0, 33, 5), (2, 57, 9), (3, 64, 4)],                # 465,156: all run in lanes
    [(1, 180, 16), (0, 21, 3)], [(0, 128, 64)], [(2, 96, 60)], [(3, 31, 7)]])
def test_mixed_iteration_equals_lanes(sizes):
    torch = need_cuda()
    ref = dpcs.Context(0, hbm_budget_bytes=1 << 30)
    c = dpcs.Context(0)
    srv = dpcs.Server(c, max_active=8, samples_per_iteration=1 << 26, quantum_samples=1 << 24)
    try:
        here, there = _resident(torch, c), _resident(torch, ref)
        slots = [srv.add_scene(h, *maps, dpcs.view_of(sc), dpcs.make_params(sc.params), sc.bounces) for sc, h, maps in here]
        outs = []
        for k, (i, side, spp) in enumerate(sizes):
            outs.append(torch.full((side, side, 3), -1.0).pin_memory())
            srv.submit(dpcs.DPCS_REQ_RELIGHT, slots[i], side, side, spp, 7 + k, torch.from_numpy(here[i][0].Ip), outs[k])
        srv.drain(60.0)
        for k, (i, side, spp) in enumerate(sizes):
            sc, h, maps = there[i]
            view = dpcs.view_of(sc.replace(Kc=np.diag([side / sc.Wc, side / sc.Hc, 1.0]).astype(np.float32) @ sc.Kc,
                                           Hc=side, Wc=side))
            Ip = torch.from_numpy(np.ascontiguousarray(sc.Ip)).cuda()
            Ic, tgt = (torch.zeros((side, side, 3), device="cuda") for _ in range(2))
            ref.render_loss_backward(h, *maps, Ip, view, dpcs.make_params(sc.params), spp, sc.bounces, 7 + k, tgt,
                                     torch.zeros(1, device="cuda"), Ic=Ic, dIp=torch.zeros_like(Ip))
            ref.sync()
            assert Ic.abs().max() > 0
            np.testing.assert_array_equal(outs[k].numpy(), Ic.cpu().numpy(), err_msg=str((i, side, spp)))
    finally:
        srv.close()
        c.close()
        ref.close()
