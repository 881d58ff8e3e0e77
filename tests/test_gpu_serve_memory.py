"""The server's memory figures count the path records of its compensation
steps, held while such requests are active, and a server whose context has a
memory budget takes none."""
import numpy as np
import pytest

from paper_2503_12174_gb300 import dpcs, scenes
from gpu_util import need_cuda

pytestmark = pytest.mark.gpu


def _run(torch, ctx_budget, sides):
    c = dpcs.Context(0, hbm_budget_bytes=ctx_budget)
    sc = scenes.corner(res=32, tex=24, bounces=3)
    maps = [torch.from_numpy(np.ascontiguousarray(x)).cuda() for x in (sc.albedo, sc.rough)]
    h = c.upload(sc.verts, sc.tris, sc.uv)
    srv = dpcs.Server(c, max_active=8)
    keep, seen = [], []
    try:
        slot = srv.add_scene(h, *maps, dpcs.view_of(sc), dpcs.make_params(sc.params), sc.bounces)
        for wave in sides:
            for side in wave:
                bufs = [torch.full((side, side, 3), 0.05).pin_memory(), torch.empty((side, side, 3)).pin_memory(),
                        torch.from_numpy(sc.Ip.copy()).pin_memory(), torch.empty(sc.Ip.shape).pin_memory()]
                keep.append(bufs)
                srv.submit(dpcs.DPCS_REQ_COMPENSATE, slot, side, side, 16, 3, bufs[2], bufs[1], target=bufs[0],
                           Ip_out=bufs[3], steps=3)
            srv.drain(60.0)
            seen.append(srv.stats())
        return seen, [(b[1].numpy().copy(), b[3].numpy().copy()) for b in keep]
    finally:
        srv.close()
        c.close()


def test_records_are_counted_and_given_back():
    """64 x 64 at 16 spp: 1,024 tiles of 64 lanes, each 24 words x 3 vertices a
    lane: 19 MB; 256 x 256: the chip's worth of tiles of 256 lanes."""
    torch = need_cuda()
    sides = [(64,), (32, 64), (256, 64)]
    free, images = _run(torch, 0, sides)
    tight, ref = _run(torch, 1 << 30, sides)
    for st in free + tight:
        assert st["memory_used"] == 0 and st["failed"] == 0
    extra = [a["memory_high_water"] - b["memory_high_water"] for a, b in zip(free, tight)]
    assert extra[0] >= 64 * 64 * 16 * 3 * 96 and extra[2] > extra[0]
    for got, want in zip(images, ref):  # the same steps in tiles and in lanes, gradients by float atomics
        np.testing.assert_allclose(got[1], want[1], rtol=0, atol=2e-3)
        np.testing.assert_allclose(got[0], want[0], rtol=2e-3, atol=2e-4)
