"""The optional scratch for path records: what a call needs and no more, none
while a stream captures, and kept for the graphs that hold its address."""
import numpy as np
import pytest

from paper_2503_12174_gb300 import dpcs, scenes
from gpu_util import need_cuda

pytestmark = pytest.mark.gpu


class _Steps:
    """A context with a corner at two image sizes and its one-trace step, FP64-accumulated."""

    def __init__(self, torch, budget=0):
        self.torch, self.c = torch, dpcs.Context(0, hbm_budget_bytes=budget)
        self.c.set_grad_accum(dpcs.DPCS_ACCUM_F64)
        sc = scenes.corner(res=32, tex=24, bounces=3, seed=5)
        self.h = self.c.upload(sc.verts, sc.tris, sc.uv)
        self.maps = [torch.from_numpy(np.ascontiguousarray(x)).cuda() for x in (sc.albedo, sc.rough, sc.Ip)]
        self.sc, self.out = sc, {}

    def step(self, res, bounces=3, stream=None):
        torch, sc = self.torch, self.sc
        if (res, bounces) not in self.out:
            self.out[res, bounces] = ([torch.zeros((res, res, 3), device="cuda") for _ in range(2)],
                                      torch.zeros(1, device="cuda"), torch.zeros_like(self.maps[2]))
        (Ic, tgt), loss, dIp = self.out[res, bounces]
        view = dpcs.view_of(sc.replace(Kc=scenes.intrinsics(res, res, 40.0), Hc=res, Wc=res))
        self.c.render_loss_backward(self.h, *self.maps, view, dpcs.make_params(sc.params), 16, bounces, 3, tgt, loss,
                                    Ic=Ic, dIp=dIp, stream=stream)
        return Ic, dIp


@pytest.mark.parametrize("principled", [False, True])
def test_small_steps_take_little_scratch(principled):
    """A 16 x 16 step fills 64 tiles: 24 (52 principled) words x 3 vertices x
    4,096 lanes and a count each, 1.2 (2.6) MB."""
    torch = need_cuda()
    used = []
    for budget in (0, 1 << 30):
        s = _Steps(torch, budget)
        try:
            if principled:
                sc = s.sc
                view = dpcs.view_of(sc.replace(Kc=scenes.intrinsics(16, 16, 40.0), Hc=16, Wc=16))
                Ic, tgt = (torch.zeros((16, 16, 3), device="cuda") for _ in range(2))
                alb, rough, Ip = s.maps
                s.c.render_loss_backward_principled(s.h, alb, rough, None, None, Ip, view, dpcs.make_params(sc.params),
                                                    16, 3, 3, tgt, torch.zeros(1, device="cuda"), Ic=Ic,
                                                    dIp=torch.zeros_like(Ip))
            else:
                s.step(16)
            s.c.sync()
            used.append(s.c.memory_used)
        finally:
            s.c.close()
    assert 0 < used[0] - used[1] <= 4096 * (3 * 4 * (52 if principled else 24) + 1) + 64 * 256


def test_capture_takes_no_scratch_and_graphs_outlive_growth():
    """A step captured before the context has records runs in lanes and
    allocates nothing; one captured with records replays after a larger step
    has replaced them.  Both give the uncaptured step's image and gradient."""
    torch = need_cuda()
    s = _Steps(torch)
    torch.cuda.synchronize()
    try:
        st = torch.cuda.Stream()
        with torch.cuda.stream(st):
            for res in (256, 64):
                s.step(res, bounces=1, stream=st)  # every other scratch buffer at its largest, but no records
            st.synchronize()
            before = s.c.memory_used
            lanes, tiles = torch.cuda.CUDAGraph(), torch.cuda.CUDAGraph()
            s.out[64, 3] = ([torch.zeros((64, 64, 3), device="cuda") for _ in range(2)], torch.zeros(1, device="cuda"),
                            torch.zeros_like(s.maps[2]))
            st.synchronize()
            with torch.cuda.graph(lanes, stream=st):
                s.step(64, stream=torch.cuda.current_stream())
            assert s.c.memory_used == before
            Ic, dIp = s.step(64, stream=st)  # records for 64 x 64
            st.synchronize()
            assert s.c.memory_used > before
            ref = Ic.clone(), dIp.clone()
            with torch.cuda.graph(tiles, stream=st):
                s.step(64, stream=torch.cuda.current_stream())
            small = s.c.memory_used
            s.step(256, stream=st)  # larger records
            st.synchronize()
            assert s.c.memory_used > small
            for graph in (lanes, tiles):
                Ic.zero_()
                dIp.zero_()
                graph.replay()
                st.synchronize()
                assert torch.equal(Ic, ref[0])
                np.testing.assert_allclose(dIp.cpu().numpy(), ref[1].cpu().numpy(), rtol=1e-5,
                                           atol=1e-6 * ref[1].abs().max().item())
    finally:
        s.c.close()
