"""Performance cases of the DPCS path tracer: what a user of the framework has
it do, through its public entry points, over the sizes it is used at.

``listed()`` names the cases, ``draw(rng)`` makes more of the same kinds and
ranges, ``prepare`` builds what a program holds before the call, ``run`` is one
pass, ``work`` counts the bytes and operations a pass cannot do without, and
``exact`` restates the result in 64-bit torch arithmetic.

Kinds:

* ``render``   -- relighting, Eq. 7: one ``Context.render``.
* ``step``     -- one gradient step of Eq. 13 (L2, gradient of Ip) or Eq. 9 (L1,
                  gradients of the maps and responses, total variation).
* ``denoised`` -- the same with the Eq. 11 filter before the loss: render with
                  kept records, filter, loss, the filter's adjoint, the kept adjoint.
* ``pose``     -- a camera-pose step: rigid move and refit, render, loss, pose adjoint.
* ``scene``    -- a mesh handed over from the host: upload (tree build), a traced
                  ray batch, a deformation (refit), the batch again, free.
* ``denoise``  -- the Eq. 11 filter and its adjoint alone.
* ``serve``    -- a batch of requests through the continuous-batching server.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

from paper_2503_12174_gb300 import dpcs, pose, scenes

RESPONSE = dict(gamma_p=(2.2, 2.4, 2.0), gain_p=1.0, gamma_c=(0.45, 0.5, 0.55), gain_c=4.0, wb=(1.1, 1.0, 0.9),
                k_proj=4.0, ks=1.0, f0=0.04)


def _case(name, kind, **kw):
    c = dict(name=name, kind=kind, mesh="corner", n_vert=0, Hc=256, Wc=256, Hp=256, Wp=256, tex=256, spp=16, bounces=3,
             rr_start=0, clip=0.0, loss="none", principled=False, radius=0, edge_spp=0, sil_spp=0, rays=0, requests=0)
    c.update(kw)
    return c


def listed():
    return [
        # the smallest call: one quad under direct light, where launches and latency are all there is
        _case("relight_plane_64", "render", mesh="plane", Hc=64, Wc=64, Hp=64, Wp=64, tex=64, spp=4, bounces=1),
        # the benchmark's headline: the interreflection corner
        _case("relight_corner_256", "render", spp=64),
        # the paper's camera and projector sizes and its second sample count, with the radiance clip of Eq. 12
        _case("relight_corner_640x360", "render", Hc=360, Wc=640, Hp=600, Wp=800, tex=512, spp=35, clip=4.0),
        # the largest render: 200k triangles, 4 bounces with Russian roulette
        _case("relight_heightfield_1024", "render", mesh="heightfield", n_vert=317, Hc=1024, Wc=1024, Hp=768, Wp=1024,
              tex=512, spp=64, bounces=4, rr_start=2),
        # the benchmark's compensation step: L2, gradient of the projector image alone
        _case("compensate_step_512", "step", Hc=512, Wc=512, Hp=512, Wp=512, tex=512, loss="l2"),
        # one pair of the scene-parameter fit at the paper's sizes: L1, gradients of maps and responses, TV
        _case("fit_step_640x360", "step", Hc=360, Wc=640, Hp=600, Wp=800, tex=512, loss="l1"),
        # the fit with metallic and normal maps
        _case("fit_principled_256", "step", loss="l1", principled=True),
        # compensation through the denoiser: the adjoint sweeps the records the render kept
        _case("compensate_denoised_512", "denoised", Hc=512, Wc=512, Hp=512, Wp=512, tex=512, loss="l2", radius=5),
        # camera-pose refinement at its default sample counts
        _case("pose_step_256", "pose", loss="l1", edge_spp=16, sil_spp=16),
        # a 200k-triangle surface arrives, is traced, deforms, is traced again
        _case("scene_heightfield_317", "scene", mesh="heightfield", n_vert=317, rays=65536),
        # the filter alone at the largest camera size
        _case("denoise_1024", "denoise", Hc=1024, Wc=1024, radius=5),
        # the serving mix: mostly relighting of several sizes, one short compensation
        _case("serve_mix_16", "serve", requests=16, spp=32),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["render", "render", "render", "step", "step", "denoised", "pose", "scene", "denoise", "serve"])
    if kind == "serve":
        return _case("", kind, requests=_log_int(rng, 2, 24), spp=_log_int(rng, 16, 64))
    if kind == "scene":
        return _case("", kind, mesh="heightfield", n_vert=_log_int(rng, 9, 317), rays=_log_int(rng, 256, 65536))
    if kind == "denoise":
        return _case("", kind, Hc=_log_int(rng, 48, 1024), Wc=_log_int(rng, 48, 1024), radius=rng.randint(2, 8))
    mesh = rng.choice(["plane", "corner", "corner", "heightfield"])
    limit = 1 << (23 if kind in ("render", "step") else 21)  # samples of one pass
    Hc, Wc = _log_int(rng, 48, 1024), _log_int(rng, 48, 1024)
    spp = _log_int(rng, 1, 96)
    if kind == "pose":
        Hc, Wc, spp = min(Hc, 384), min(Wc, 384), min(spp, 16)
    spp = max(1, min(spp, limit // (Hc * Wc)))
    bounces = 1 if mesh == "plane" else rng.randint(2, 4)
    if kind == "denoised":
        spp = min(spp, 32)
    return _case("", kind, mesh=mesh, n_vert=_log_int(rng, 17, 317) if mesh == "heightfield" else 0, Hc=Hc, Wc=Wc,
                 Hp=_log_int(rng, 64, 800), Wp=_log_int(rng, 64, 1024), tex=_log_int(rng, 33, 512), spp=spp,
                 bounces=bounces, rr_start=2 if mesh == "heightfield" and rng.random() < 0.5 else 0,
                 clip=4.0 if rng.random() < 0.25 else 0.0,
                 loss="none" if kind == "render" else ("l1" if kind == "pose" else rng.choice(["l1", "l2"])),
                 principled=mesh == "corner" and kind in ("render", "step", "denoised") and rng.random() < 0.3,
                 radius=rng.randint(2, 6) if kind == "denoised" else 0,
                 edge_spp=rng.choice([4, 16]) if kind == "pose" else 0, sil_spp=4 if kind == "pose" else 0)


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
@functools.lru_cache(maxsize=1)
def _corner():
    return scenes.corner_mesh()


def _mesh(case, rng):
    if case["mesh"] == "corner":
        return _corner()
    if case["mesh"] == "plane":
        return (np.array([[-1, -1, 1], [1, -1, 1], [1, 1, 1], [-1, 1, 1]], np.float32),
                np.array([[0, 1, 2], [0, 2, 3]], np.int32), np.array([[0, 0], [1, 0], [1, 1], [0, 1]], np.float32))
    return scenes.heightfield_mesh(rng, n_vert=case["n_vert"])


def _blobs(rng, H, W):
    """A projector image or photograph: smooth coloured blobs in [0, 1]."""
    y, x = (np.arange(H) + 0.5) / H, (np.arange(W) + 0.5) / W
    c, s = rng.random((8, 2)), 0.05 + 0.25 * rng.random((8, 1))
    gy, gx = np.exp(-(y - c[:, :1]) ** 2 / (2 * s * s)), np.exp(-(x - c[:, 1:]) ** 2 / (2 * s * s))
    img = np.einsum("by,bx,bc->yxc", gy, gx, rng.random((8, 3)), optimize=True)
    return np.ascontiguousarray(img / img.max(), np.float32)


def _noise(rng, n, lo, hi):
    return (lo + (hi - lo) * scenes.smooth_noise(rng, n, n)).astype(np.float32)


def _inputs(case, seed):
    """Host arrays of a rendering case, from the seed alone."""
    rng = np.random.default_rng([seed, 17])
    verts, tris, uv = _mesh(case, rng)
    fov_c, fov_p = {"plane": (40.0, 40.0), "corner": (40.0, 45.0), "heightfield": (62.0, 50.0)}[case["mesh"]]
    if case["mesh"] == "corner":
        Rp, tp = scenes.look_at((0.25, -0.15, 0.0), (-0.05, 0.1, 1.3))
    elif case["mesh"] == "plane":
        Rp, tp = np.eye(3, dtype=np.float32), np.array([-0.3, 0, 0], np.float32)
    else:
        Rp, tp = scenes.look_at((0.3, -0.2, 0.0), (0.0, 0.0, 1.5))
    n = case["tex"]
    albedo = np.ascontiguousarray(np.stack([_noise(rng, n, 0.2, 0.9) for _ in range(3)], -1))
    rough = _noise(rng, n, 0.1, 0.8)
    d = dict(verts=verts, tris=tris, uv=uv, albedo=albedo, rough=rough, Ip=_blobs(rng, case["Hp"], case["Wp"]),
             Kc=scenes.intrinsics(case["Wc"], case["Hc"], fov_c), Kp=scenes.intrinsics(case["Wp"], case["Hp"], fov_p),
             Rp=Rp, tp=tp)
    if case["loss"] != "none":
        d["target"] = 0.7 * _blobs(rng, case["Hc"], case["Wc"])
    if case["principled"]:
        d["metallic"], d["normal"] = scenes.principled_maps(rng, n, n)
    return d


def _params(case):
    p = dict(RESPONSE, rr_start=case["rr_start"], rr_q=0.75 if case["rr_start"] else 1.0, clip=case["clip"])
    if case["mesh"] == "plane":
        p.update(ks=0.0)
    return scenes.Params(**p)


def _rays(case, seed, n):
    """Rays from around the camera into the surface."""
    rng = np.random.default_rng([seed, 23])
    o = rng.uniform(-0.2, 0.2, (n, 3)).astype(np.float32)
    d = rng.normal(0.0, 0.35, (n, 3)).astype(np.float32)
    d[:, 2] = 1.0
    d /= np.linalg.norm(d, axis=1, keepdims=True).astype(np.float32)
    return o, d


def _deformed(verts):
    v = verts.copy()
    v[:, 2] += 0.03 * np.sin(5.0 * verts[:, 0]) * np.cos(4.0 * verts[:, 1])
    return v


def _filter_inputs(case, seed):
    """A noisy image, guide features of a piecewise smooth scene, and a gradient."""
    g = torch.Generator().manual_seed(seed)
    H, W = case["Hc"], case["Wc"]
    rng = np.random.default_rng([seed, 29])
    img = torch.from_numpy(_blobs(rng, H, W)) * (0.6 + 0.8 * torch.rand((H, W, 3), generator=g))
    y, x = torch.meshgrid(torch.arange(H) / H, torch.arange(W) / W, indexing="ij")
    side = (x + 0.3 * y > 0.6).float()[..., None]
    alb = torch.from_numpy(_blobs(rng, H, W))
    nrm = torch.nn.functional.normalize(torch.stack([0.4 * torch.sin(7 * x), 0.4 * torch.cos(9 * y), -torch.ones_like(x)],
                                                    -1) + side * torch.tensor([1.0, 0.0, 0.3]), dim=-1)
    guide = torch.cat([alb, nrm, (1.0 + 0.5 * x + 0.2 * y)[..., None] + 0.4 * side, torch.ones((H, W, 1))], -1)
    return img, guide, torch.randn((H, W, 3), generator=g)


def _requests(case, seed):
    """The serving mix: the case fixes the camera sides and sample counts (log-uniform) and which request
    compensates, the seed the images and sample streams."""
    shape, rng = np.random.default_rng([case["requests"], case["spp"]]), np.random.default_rng([seed, 31])
    out = []
    for i in range(case["requests"]):
        slot, side, f = int(shape.integers(2)), int(64 * shape.integers(2, 9)), float(2 ** shape.uniform(-1, 1))
        comp = i == case["requests"] // 2
        side = 128 if comp else side
        out.append(dict(comp=comp, slot=slot, side=side, spp=16 if comp else max(1, int(case["spp"] * f)),
                        seed=int(rng.integers(1 << 30)), Ip=_blobs(rng, 256, 256) if slot else _blobs(rng, 64, 64),
                        target=0.7 * _blobs(rng, side, side) if comp else None))
    return out


def _serve_scenes(seed):
    plane = _case("", "render", mesh="plane", Hc=64, Wc=64, Hp=64, Wp=64, tex=64, bounces=1)
    corner = _case("", "render")
    return [(c, _inputs(c, seed + k)) for k, c in enumerate((plane, corner))]


# ---------------------------------------------------------------------------
# state and one pass
# ---------------------------------------------------------------------------
class State:
    pass


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def _view(d, case):
    return dpcs.make_view(d["Kc"], case["Hc"], case["Wc"], d["Kp"], d["Rp"], d["tp"], case["Hp"], case["Wp"])


def prepare(case, seed):
    s = State()
    s.case, s.seed, s.ctx = case, seed, dpcs.Context(0)
    kind = case["kind"]
    if kind == "denoise":
        s.img, s.guide, s.dD = (t.cuda() for t in _filter_inputs(case, seed))
        s.prm = dpcs.make_denoise_params(radius=case["radius"])
        return s
    if kind == "scene":
        s.verts, s.tris, s.uv = _mesh(case, np.random.default_rng([seed, 17]))
        s.moved = _deformed(s.verts)
        s.o, s.d = (_dev(a) for a in _rays(case, seed, case["rays"]))
        return s
    if kind == "serve":
        s.server = dpcs.Server(s.ctx)
        s.keep = []
        for c, d in _serve_scenes(seed):
            h = s.ctx.upload(d["verts"], d["tris"], d["uv"])
            alb, rough = _dev(d["albedo"]), _dev(d["rough"])
            s.server.add_scene(h, alb, rough, _view(d, c), dpcs.make_params(_params(c)), c["bounces"])
            s.keep.append((alb, rough))
        s.reqs = []
        for r in _requests(case, seed):
            pin = {k: torch.from_numpy(r[k]).pin_memory() for k in ("Ip", "target") if r[k] is not None}
            s.reqs.append((r, pin, torch.empty((r["side"], r["side"], 3)).pin_memory(),
                           torch.empty(tuple(r["Ip"].shape)).pin_memory() if r["comp"] else None))
        return s
    d = _inputs(case, seed)
    s.h = s.ctx.upload(d["verts"], d["tris"], d["uv"])
    s.view, s.params = _view(d, case), dpcs.make_params(_params(case))
    s.alb, s.rough, s.Ip = _dev(d["albedo"]), _dev(d["rough"]), _dev(d["Ip"])
    s.met, s.nrm = (_dev(d[k]) if case["principled"] else None for k in ("metallic", "normal"))
    s.Ic = torch.empty((case["Hc"], case["Wc"], 3), device="cuda")
    s.Ec = torch.empty_like(s.Ic)
    if kind == "render":
        return s
    s.target, s.loss = _dev(d["target"]), torch.zeros(1, device="cuda")
    s.dIc = torch.empty_like(s.Ic)
    s.scale = 1.0 if case["loss"] == "l2" else 1.0 / s.Ic.numel()
    if kind == "pose":
        s.wrench = torch.zeros((3, 6), dtype=torch.float64, device="cuda")
        s.R, s.t = pose.pose_of([0.004, -0.003, 0.002, 0.003, -0.002, 0.004])
        s.posed = pose.posed_view(s.view, s.R, s.t)
        return s
    if kind == "denoised":
        s.guide = torch.empty((case["Hc"], case["Wc"], 8), device="cuda")
        s.prm = dpcs.make_denoise_params(radius=case["radius"])
        s.D, s.dD = torch.empty_like(s.Ic), torch.empty_like(s.Ic)
        s.wsum = torch.empty((case["Hc"], case["Wc"]), device="cuda")
    if case["loss"] == "l2":
        s.grads = {"dIp": torch.zeros_like(s.Ip)}
    else:
        s.grads = {"dAlbedo": torch.zeros_like(s.alb), "dRough": torch.zeros_like(s.rough),
                   "dParams": torch.zeros(11, device="cuda")}
        s.tv = torch.zeros(2, device="cuda")
        if case["principled"]:
            s.grads.update(dMetallic=torch.zeros_like(s.met), dNormal=torch.zeros_like(s.nrm))
    return s


TV_WEIGHT = 1e-5


def run(s):
    case, c = s.case, s.ctx
    kind, spp, b = case["kind"], case["spp"], case["bounces"]
    if kind == "denoise":
        D, wsum = c.denoise(s.img, s.guide, s.prm)
        return D, wsum, c.denoise_backward(s.dD, s.guide, wsum, s.prm)
    if kind == "scene":
        h = c.upload(s.verts, s.tris, s.uv)
        t0, tri0 = c.trace(h, s.o, s.d)
        c.update(h, s.moved)
        t1, tri1 = c.trace(h, s.o, s.d)
        c.free(h)
        return t0, tri0, t1, tri1
    if kind == "serve":
        for r, pin, Ic, Ip_out in s.reqs:
            s.server.submit(dpcs.DPCS_REQ_COMPENSATE if r["comp"] else dpcs.DPCS_REQ_RELIGHT, r["slot"], r["side"],
                            r["side"], r["spp"], r["seed"], pin["Ip"], Ic, target=pin.get("target"), Ip_out=Ip_out,
                            steps=4 if r["comp"] else 0)
        s.server.drain()
        return [x for _, _, Ic, Ip_out in s.reqs for x in (Ic, Ip_out) if x is not None]
    tex = (s.alb, s.rough, s.met, s.nrm) if case["principled"] else (s.alb, s.rough)
    render = c.render_principled if case["principled"] else c.render
    if kind == "render":
        render(s.h, *tex, s.Ip, s.view, s.params, spp, b, s.seed, Ic=s.Ic, Ec=s.Ec)
        return s.Ic, s.Ec
    if kind == "pose":
        c.transform(s.h, s.R, s.t)
        s.wrench.zero_()
        c.render(s.h, s.alb, s.rough, s.Ip, s.posed, s.params, spp, b, s.seed, Ic=s.Ic, Ec=s.Ec)
        c.l1_loss(s.Ic, s.target, s.dIc, s.loss, scale=s.scale)
        c.pose_backward(s.h, s.alb, s.rough, s.Ip, s.posed, s.params, spp, b, pose.adjoint_key(s.seed), s.Ec, s.Ic,
                        s.dIc, case["edge_spp"], case["sil_spp"], wrench=s.wrench)
        return s.Ic, s.loss, s.wrench
    for g in s.grads.values():
        g.zero_()
    if kind == "step":
        f = c.render_loss_backward_principled if case["principled"] else c.render_loss_backward
        f(s.h, *tex, s.Ip, s.view, s.params, spp, b, s.seed, s.target, s.loss, loss_kind=int(case["loss"] == "l1"),
          scale=s.scale, Ic=s.Ic, Ec=s.Ec, **s.grads)
    else:
        c.gbuffer(s.h, s.alb, s.rough, s.view, guide=s.guide)
        render(s.h, *tex, s.Ip, s.view, s.params, spp, b, s.seed, Ic=s.Ic, Ec=s.Ec, keep=True)
        c.denoise(s.Ic, s.guide, s.prm, out=s.D, wsum=s.wsum)
        if case["loss"] == "l2":
            c.l2_loss(s.D, s.target, s.dD, s.loss)
        else:
            c.l1_loss(s.D, s.target, s.dD, s.loss, scale=s.scale)
        s.dIc.zero_()
        c.denoise_backward(s.dD, s.guide, s.wsum, s.prm, dIc=s.dIc)
        back = c.render_backward_principled if case["principled"] else c.render_backward
        back(s.h, *tex, s.Ip, s.view, s.params, spp, b, s.seed, s.Ec, s.Ic, s.dIc, kept=True, **s.grads)
    if case["loss"] == "l1":
        c.tv_loss(s.alb, s.grads["dAlbedo"], s.tv[0:1], TV_WEIGHT)
        c.tv_loss(s.rough, s.grads["dRough"], s.tv[1:2], TV_WEIGHT)
        return [s.Ic, s.loss, s.tv, *s.grads.values()]
    return [s.Ic, s.loss, *s.grads.values()]


# ---------------------------------------------------------------------------
# the work a pass cannot do without
# ---------------------------------------------------------------------------
def _triangles(case):
    return {"plane": 2, "corner": 1026, "heightfield": 2 * (case["n_vert"] - 1) ** 2}[case["mesh"]]


def _path_flops(case, samples):
    """Per vertex: one box descent to the hit and one to the projector (26 operations a node over log2 T
    levels), two triangle tests (46 each), the vertex (140), its light (160) and the continuation (230)."""
    levels = max(1.0, math.log2(_triangles(case)))
    vertices = 1.0 if case["bounces"] == 1 else 2.0  # paths end on misses, below the surface and by roulette
    return samples * (27 + vertices * (2 * 26 * levels + 92 + 140 + 160 + 230))


def work(case):
    kind = case["kind"]
    npix, np_, nt, T = case["Hc"] * case["Wc"], case["Hp"] * case["Wp"], case["tex"] ** 2, _triangles(case)
    if kind == "denoise":  # image, guide in; image, weights out; and the adjoint's gradient in and out
        taps = (2 * case["radius"] + 1) ** 2
        return {"bytes": npix * (12 + 32 + 12 + 4 + 12 + 12), "flops": 2 * npix * taps * 32}
    if kind == "scene":  # mesh in, nodes and triangles out; new vertices in, nodes and triangles out; rays, hits
        V, n = case["n_vert"] ** 2, case["rays"]
        return {"bytes": V * 20 + T * 12 + T * (64 + 48 + 24) + V * 12 + T * (64 + 48) + n * (24 + 16),
                "flops": T * 200 + 2 * n * (26 * max(1.0, math.log2(T)) + 92)}
    if kind == "serve":
        b = f = 0.0
        for r in _requests(case, 0):
            c = _case("", "render", mesh="corner" if r["slot"] else "plane", bounces=3 if r["slot"] else 1)
            n = r["side"] ** 2
            b += 2 * r["Ip"].size * 4 + n * 12
            f += _path_flops(c, n * r["spp"]) * (8 if r["comp"] else 1)
        return {"bytes": b, "flops": f}
    maps = 12 + 4 + (16 if case["principled"] else 0)
    scene = T * (48 + 24 + 64)
    by, fl = npix * 24 + np_ * 12 + nt * maps + scene, _path_flops(case, npix * case["spp"])
    if kind == "render":
        return {"bytes": by, "flops": fl}
    if kind == "pose":
        edges = 4 * npix * case["edge_spp"]
        return {"bytes": by + npix * 24 + 2 * scene, "flops": 2 * fl + _path_flops(case, edges)}
    by += npix * 12 + (np_ * 12 if case["loss"] == "l2" else nt * (2 * maps + 16))
    fl += npix * case["spp"] * 2 * 104
    if kind == "denoised":
        f = work(_case("", "denoise", Hc=case["Hc"], Wc=case["Wc"], radius=case["radius"]))
        by, fl = by + f["bytes"], fl + f["flops"] + npix * (27 + 140)
    return {"bytes": by, "flops": fl}


# ---------------------------------------------------------------------------
# the results in 64-bit torch arithmetic
# ---------------------------------------------------------------------------
MAX_TESTS = 6e10  # ray-triangle pairs of a brute-force pass that take a few seconds; more would not fit 20 s
_F = torch.float64


def _uniforms(seed, pix, s, b):
    """Philox4x32-10 (Salmon et al., SC'11), counter (pix, s, b, 0): four 24-bit uniforms."""
    M = 0xFFFFFFFF
    k0, k1 = seed & M, (seed >> 32) & M
    c = [pix, s, torch.full_like(pix, b), torch.zeros_like(pix)]
    for _ in range(10):
        p0, p1 = c[0] * 0xD2511F53, c[2] * 0xCD9E8D57  # wraps modulo 2^64
        c = [((p1 >> 32) & M) ^ c[1] ^ k0, p1 & M, ((p0 >> 32) & M) ^ c[3] ^ k1, p0 & M]
        k0, k1 = (k0 + 0x9E3779B9) & M, (k1 + 0xBB67AE85) & M
    return [(x >> 8).to(_F) * 2.0 ** -24 for x in c]


def _dot(a, b):
    return (a * b).sum(-1, keepdim=True)


def _unit(a):
    return a / _dot(a, a).sqrt()


class _Geometry:
    """Brute-force ray casting: with m = o x d every barycentric numerator is linear in (d, m)."""

    def __init__(self, verts, tris, uv):
        v = torch.from_numpy(verts).cuda().to(_F)
        f = torch.from_numpy(tris).cuda().long()
        self.v0, self.e1, self.e2 = v[f[:, 0]], v[f[:, 1]] - v[f[:, 0]], v[f[:, 2]] - v[f[:, 0]]
        self.n = torch.linalg.cross(self.e1, self.e2)
        z = torch.zeros_like(self.n)
        self.Md = torch.cat([-self.n, z], 1).T.contiguous()
        self.Mu = torch.cat([-torch.linalg.cross(self.e2, self.v0), self.e2], 1).T.contiguous()
        self.Mv = torch.cat([-torch.linalg.cross(self.v0, self.e1), -self.e1], 1).T.contiguous()
        self.nv0 = (self.n * self.v0).sum(1)
        self.uv = torch.from_numpy(uv).cuda().to(_F)[f]

    def _all(self, o, d):
        ray = torch.cat([d, torch.linalg.cross(o, d)], 1)
        inv = 1.0 / (ray @ self.Md)
        u, v = (ray @ self.Mu) * inv, (ray @ self.Mv) * inv
        t = (o @ self.n.T - self.nv0) * inv
        return torch.where((u >= 0) & (v >= 0) & (u + v <= 1) & (t > 0), t, math.inf)

    def closest(self, o, d):
        step = max(1, 1 << 26 >> max(0, self.n.shape[0] - 1).bit_length())
        parts = [self._all(o[i:i + step], d[i:i + step]).min(1) for i in range(0, max(1, len(o)), step)]
        t, k = torch.cat([p.values for p in parts]), torch.cat([p.indices for p in parts])
        ray = torch.cat([d, torch.linalg.cross(o, d)], 1)
        det = (ray * self.Md.T[k]).sum(1)
        return t, k, (ray * self.Mu.T[k]).sum(1) / det, (ray * self.Mv.T[k]).sum(1) / det


def _bilinear(img, x, y):
    """Texel centres at i + 1/2, clamped to the edge."""
    H, W = img.shape[:2]
    x, y = (x - 0.5).clamp(-1, W), (y - 0.5).clamp(-1, H)
    x0, y0 = x.floor(), y.floor()
    fx, fy = x - x0, y - y0
    xa, xb = x0.long().clamp(0, W - 1), (x0.long() + 1).clamp(0, W - 1)
    ya, yb = y0.long().clamp(0, H - 1), (y0.long() + 1).clamp(0, H - 1)
    flat = img.reshape(H * W, -1)
    return (flat[ya * W + xa] * ((1 - fx) * (1 - fy))[:, None] + flat[ya * W + xb] * (fx * (1 - fy))[:, None] +
            flat[yb * W + xa] * ((1 - fx) * fy)[:, None] + flat[yb * W + xb] * (fx * fy)[:, None])


def _basis(n):
    """Duff et al., JCGT 2017, with the seam at n.z = -1/pi."""
    x, y, z = n.unbind(-1)
    sg = torch.where(z >= -1.0 / math.pi, 1.0, -1.0).to(_F)
    a = -1.0 / (sg + z)
    return (torch.stack([1 + sg * x * x * a, sg * x * y * a, -sg * x], -1),
            torch.stack([x * y * a, sg + y * y * a, -y], -1))


def _ggx(n, h, a):
    a2, c = a * a, torch.linalg.cross(n, h)
    t = _dot(c, c) + a2 * _dot(n, h) ** 2
    return a2 / (math.pi * t * t)


def _masking(c, a):
    return 2 * c / (c + (a * a + (1 - a * a) * c * c).sqrt())


class _Tracer:
    """The path tracer of Eqs. 1-6 and 10 (Lambert + GGX, or the metallic
    workflow with a normal map) with detached sampling."""

    def __init__(self, case, d, seed, prm):
        self.case, self.seed, self.p = case, seed, prm
        self.g = _Geometry(d["verts"], d["tris"], d["uv"])
        t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda().to(_F)
        self.Kci, self.Kp, self.Rp, self.tp = t(d["Kc"]).inverse(), t(d["Kp"]), t(d["Rp"]), t(d["tp"])
        self.cp = -self.Rp.T @ self.tp
        self.Ip, self.alb, self.rough = t(d["Ip"]), t(d["albedo"]), t(d["rough"])
        nt = self.rough.shape
        self.met = t(d["metallic"]) if "metallic" in d else torch.zeros(nt, dtype=_F, device="cuda")
        self.nrm = t(d["normal"]) if "normal" in d else None
        self.gp, self.Gp = t(np.array(prm.gamma_p)), t(np.array(prm.gain_p))
        self.Ep = torch.where(self.Ip > 0, self.Gp * self.Ip.clamp_min(1e-300) ** self.gp, 0.0)
        self.ks, self.f0 = float(np.float32(prm.ks)), float(np.float32(prm.f0))

    def surface(self, k, u, v, d):
        g = self.g
        x = g.v0[k] + g.e1[k] * u[:, None] + g.e2[k] * v[:, None]
        n = _unit(g.n[k])
        n = torch.where(_dot(n, d) > 0, -n, n)
        c = g.uv[k]
        st = c[:, 0] * (1 - u - v)[:, None] + c[:, 1] * u[:, None] + c[:, 2] * v[:, None]
        H, W = self.rough.shape
        return x, n, st[:, 0] * W, st[:, 1] * H

    def brdf(self, ns, wo, wi, rho, r, m):
        co, ci = _dot(ns, wo), _dot(ns, wi)
        on = (co > 0) & (ci > 0)
        co, ci = torch.where(on, co, 1.0), torch.where(on, ci, 1.0)
        a = r.clamp(0.01, 1.0) ** 2
        h = _unit(wo + wi)
        S = self.ks * _ggx(ns, h, a) * _masking(ci, a) * _masking(co, a) / (4 * ci * co)
        F0 = (1 - m) * self.f0 + m * rho
        F = F0 + (1 - F0) * (1 - _dot(wo, h)).clamp_min(0) ** 5
        return torch.where(on, (1 - m) * rho / math.pi + S * F, 0.0)

    def sample(self, ns, wo, r, u):
        """The lobe's direction and pdf: cosine hemisphere, or visible normals (Heitz, JCGT 2018)."""
        T, B = _basis(ns)
        ps = 0.5 if self.ks > 0 else 0.0
        c, s = torch.cos(2 * math.pi * u[2]), torch.sin(2 * math.pi * u[2])
        rr = u[1].sqrt()
        lam = torch.stack([rr * c, rr * s, (1 - u[1]).clamp_min(0).sqrt()], -1)
        a = r.clamp(0.01, 1.0) ** 2
        wl = torch.cat([_dot(wo, T), _dot(wo, B), _dot(wo, ns)], 1)
        Vh = _unit(torch.cat([a * wl[:, :2], wl[:, 2:]], 1))
        l2 = Vh[:, :1] ** 2 + Vh[:, 1:2] ** 2
        T1 = torch.where(l2 > 0, torch.cat([-Vh[:, 1:2], Vh[:, :1], torch.zeros_like(l2)], 1) / l2.clamp_min(1e-300).sqrt(),
                         torch.tensor([1.0, 0.0, 0.0], dtype=_F, device="cuda"))
        T2 = torch.linalg.cross(Vh, T1)
        t1, t2, w = (rr * c)[:, None], (rr * s)[:, None], 0.5 * (1 + Vh[:, 2:])
        t2 = (1 - w) * (1 - t1 * t1).clamp_min(0).sqrt() + w * t2
        Nh = T1 * t1 + T2 * t2 + Vh * (1 - t1 * t1 - t2 * t2).clamp_min(0).sqrt()
        Ne = _unit(torch.cat([a * Nh[:, :2], Nh[:, 2:].clamp_min(0)], 1))
        spec = Ne * (2 * _dot(wl, Ne)) - wl
        l = torch.where((u[0] >= ps)[:, None], lam, spec)
        wi = T * l[:, :1] + B * l[:, 1:2] + ns * l[:, 2:]
        ci, co = _dot(ns, wi), _dot(ns, wo)
        pdf = (1 - ps) * ci / math.pi
        if ps > 0:
            h = _unit(wo + wi)
            pdf = pdf + ps * _masking(co, a) * _ggx(ns, h, a) / (4 * co)
        ok = (ci > 0) & (co > 0) & (pdf > 0)
        return wi, torch.where(ok, pdf, 1.0), ok[:, 0]

    def radiance(self, pix, s, tex, mat, Ep):
        """Path radiance (N, 3) of samples s of pixels pix; differentiable in tex, mat and Ep."""
        case, p, N = self.case, self.p, len(pix)
        u = _uniforms(self.seed, pix, s, 0)
        xy = torch.stack([(pix % case["Wc"]).to(_F) + u[0], (pix // case["Wc"]).to(_F) + u[1], torch.ones_like(u[0])], -1)
        d, o = _unit(xy @ self.Kci.T), torch.zeros((N, 3), dtype=_F, device="cuda")
        L = torch.zeros((N, 3), dtype=_F, device="cuda")
        beta, live = torch.ones_like(L), torch.arange(N, device="cuda")
        eps, Hp, Wp = float(np.float32(1e-4)), case["Hp"], case["Wp"]
        for b in range(1, case["bounces"] + 1):
            t, k, u_, v_ = self.g.closest(o, d)
            hit = torch.isfinite(t)
            live, k, u_, v_, d, beta = live[hit], k[hit], u_[hit], v_[hit], d[hit], beta[hit]
            x, n, tx, ty = self.surface(k, u_, v_, d)
            q = _bilinear(tex, tx, ty)
            rho, r, wo = q[:, :3], q[:, 3:], -d
            m, ns = torch.zeros_like(r), n
            if mat is not None:
                q = _bilinear(mat, tx, ty)
                m, nm = q[:, :1], 2 * q[:, 1:] - 1
                e1, e2, c = self.g.e1[k], self.g.e2[k], self.g.uv[k]
                d1, d2 = c[:, 1] - c[:, 0], c[:, 2] - c[:, 0]
                det = (d1[:, 0] * d2[:, 1] - d2[:, 0] * d1[:, 1])[:, None]
                dpdu = (e1 * d2[:, 1:] - e2 * d1[:, 1:]) / det
                T = dpdu - n * _dot(n, dpdu)
                good = (det != 0) & (_dot(T, T) > 1e-12 * _dot(dpdu, dpdu))
                T = torch.where(good, _unit(torch.where(good, T, torch.ones_like(T))), _basis(n)[0])
                ns = _unit(T * nm[:, :1] + torch.linalg.cross(n, T) * nm[:, 1:2] + n * nm[:, 2:])
            # next-event estimation to the pinhole projector
            X = x @ self.Rp.T + self.tp
            w = X @ self.Kp.T
            up, vp = w[:, 0] / w[:, 2], w[:, 1] / w[:, 2]
            v = self.cp - x
            r2 = _dot(v, v)
            wp = v / r2.sqrt()
            cs = _dot(ns, wp)
            lit = ((w[:, 2] > 0) & (X[:, 2] > 0) & (up >= 0) & (up < Wp) & (vp >= 0) & (vp < Hp) & (cs[:, 0] > 0) &
                   (_dot(n, wp)[:, 0] > 0))
            so = x + n * eps
            sv = self.cp - so
            sd = _dot(sv, sv).sqrt()
            i = lit.nonzero()[:, 0]
            blocked = self.g.closest(so[i], (sv / sd)[i])[0] < sd[i, 0] - eps
            i = i[~blocked]
            G = p.k_proj * (X[:, 2:] / _dot(X, X).sqrt())[i] * cs[i] / r2[i]
            f = self.brdf(ns[i], wo[i], wp[i], rho[i], r[i], m[i])
            c = beta[i] * f * _bilinear(Ep, up[i], vp[i]) * G
            L = L.index_add(0, live[i], c.clamp(max=p.clip) if p.clip > 0 else c)
            if b == case["bounces"]:
                break
            with torch.no_grad():
                u = _uniforms(self.seed, pix[live], s[live], b)
                wi, pdf, ok = self.sample(ns, wo, r, u)
                ok &= _dot(n, wi)[:, 0] > 0
                rrq = 1.0
                if p.rr_start > 0 and b >= p.rr_start:
                    rrq = float(np.float32(p.rr_q))
                    ok &= u[3] < rrq
                i = ok.nonzero()[:, 0]
            beta = beta[i] * self.brdf(ns[i], wo[i], wi[i], rho[i], r[i], m[i]) * (_dot(ns[i], wi[i]) / (pdf[i] * rrq))
            live, o, d = live[i], so[i], wi[i]
        return L

    def _chunks(self):
        npix, spp = self.case["Hc"] * self.case["Wc"], self.case["spp"]
        step = max(1, (1 << 20) // spp)
        for a in range(0, npix, step):
            n = min(step, npix - a)
            pix = torch.arange(a, a + n, device="cuda").repeat_interleave(spp)
            yield a, n, pix, torch.arange(spp, device="cuda").repeat(n)

    def _maps(self):
        tex = torch.cat([self.alb, self.rough[..., None]], -1)
        return tex, None if self.nrm is None else torch.cat([self.met[..., None], self.nrm], -1)

    @torch.no_grad()
    def image(self):
        tex, mat = self._maps()
        spp = self.case["spp"]
        out = [self.radiance(pix, s, tex, mat, self.Ep).view(n, spp, 3).mean(1) for _, n, pix, s in self._chunks()]
        return torch.cat(out).view(self.case["Hc"], self.case["Wc"], 3)

    def response(self, Ec):
        """Ic of Eq. 5 and the leaves (gamma_c, Gc, wb) it depends on."""
        leaves = [torch.tensor(v, dtype=torch.float32, device="cuda").to(_F).requires_grad_() for v in
                  (self.p.gamma_c, self.p.gain_c, self.p.wb)]
        a = leaves[1] * leaves[2] * Ec
        return torch.where(a > 0, a.clamp_min(1e-300) ** leaves[0], 0.0), leaves

    def gradients(self, dEc):
        """dLoss/d(Ip, tex, mat, gamma_p, Gp) from dLoss/dEc."""
        tex, mat = self._maps()
        leaves = [t.detach().clone().requires_grad_() for t in (tex, self.Ep)] + \
            ([mat.detach().clone().requires_grad_()] if mat is not None else [])
        g = (dEc / self.case["spp"]).view(-1, 3)
        for a, n, pix, s in self._chunks():
            L = self.radiance(pix, s, leaves[0], leaves[2] if mat is not None else None, leaves[1])
            if L.requires_grad:
                L.backward(g[a:a + n].repeat_interleave(self.case["spp"], 0))
        Ip, gp, Gp = (t.detach().clone().requires_grad_() for t in (self.Ip, self.gp, self.Gp))
        Ep = torch.where(Ip > 0, Gp * Ip.clamp_min(1e-300) ** gp, 0.0)
        dEp = leaves[1].grad if leaves[1].grad is not None else torch.zeros_like(self.Ep)
        Ep.backward(dEp)
        zero = [torch.zeros_like(t) if t.grad is None else t.grad for t in leaves]
        return Ip.grad, zero[0], zero[2] if mat is not None else None, gp.grad, Gp.grad

    @torch.no_grad()
    def guide(self):
        pix = torch.arange(self.case["Hc"] * self.case["Wc"], device="cuda")
        xy = torch.stack([pix % self.case["Wc"] + 0.5, pix // self.case["Wc"] + 0.5, torch.ones_like(pix)], -1).to(_F)
        d = _unit(xy @ self.Kci.T)
        t, k, u, v = self.g.closest(torch.zeros_like(d), d)
        x, n, tx, ty = self.surface(k, u, v, d)
        q = torch.cat([_bilinear(self.alb, tx, ty), n, t[:, None], torch.ones_like(t)[:, None]], 1)
        return torch.where(torch.isfinite(t)[:, None], q, 0.0).view(self.case["Hc"], self.case["Wc"], 8)


@torch.no_grad()
def _gather(img, guide, radius):
    """sum_q w(p, q) img(q) and sum_q w(p, q) of Eq. 11 with the default widths."""
    H, W = img.shape[:2]
    k = [0.5 / float(np.float32(s)) ** 2 for s in (2.0, 0.1, 0.3, 0.1)]
    num, den = torch.zeros_like(img), torch.zeros((H, W), dtype=_F, device="cuda")
    for dy in range(-radius, radius + 1):
        for dx in range(-radius, radius + 1):
            y0, y1, x0, x1 = max(0, -dy), H - max(0, dy), max(0, -dx), W - max(0, dx)
            if y0 >= y1 or x0 >= x1:
                continue
            q = (slice(y0 + dy, y1 + dy), slice(x0 + dx, x1 + dx))
            e = (guide[y0:y1, x0:x1] - guide[q])[..., :7] ** 2
            w = torch.exp(-((dx * dx + dy * dy) * k[0] + e[..., :3].sum(-1) * k[1] + e[..., 3:6].sum(-1) * k[2] +
                            e[..., 6] * k[3]))
            num[y0:y1, x0:x1] += w[..., None] * img[q]
            den[y0:y1, x0:x1] += w
    return num, den


def _tv(m, weight):
    m = m.detach().clone().requires_grad_()
    loss = weight * ((m[1:] - m[:-1]).abs().sum() + (m[:, 1:] - m[:, :-1]).abs().sum())
    loss.backward()
    return loss.detach(), m.grad


def _tests(case):
    return case["Hc"] * case["Wc"] * case["spp"] * case["bounces"] * 2 * _triangles(case)


def exact(case, seed):
    kind = case["kind"]
    if kind == "denoise":
        img, guide, dD = (t.cuda().to(_F) for t in _filter_inputs(case, seed))
        num, den = _gather(img, guide, case["radius"])
        return num / den[..., None], den, _gather(dD / den[..., None], guide, case["radius"])[0]
    if kind == "scene":  # distances; the hit triangle of a ray through an edge is a matter of rounding
        if 2.0 * case["rays"] * _triangles(case) > MAX_TESTS:
            return None
        verts, tris, uv = _mesh(case, np.random.default_rng([seed, 17]))
        o, d = (_dev(a).to(_F) for a in _rays(case, seed, case["rays"]))
        t0, t1 = (_Geometry(v, tris, uv).closest(o, d)[0] for v in (verts, _deformed(verts)))
        return t0, None, t1, None
    if kind == "serve":  # the relit images; a few Adam steps amplify any rounding of a gradient's sign
        parts = _serve_scenes(seed)
        out = []
        for r in _requests(case, seed):
            if r["comp"]:
                out += [None, None]
                continue
            c, d = parts[r["slot"]]
            k = np.array([[r["side"] / c["Wc"]], [r["side"] / c["Hc"]], [1.0]], np.float32)
            c = dict(c, Hc=r["side"], Wc=r["side"], spp=r["spp"])
            if _tests(c) > MAX_TESTS / 8:
                out.append(None)
                continue
            tr = _Tracer(c, dict(d, Kc=d["Kc"] * k, Ip=r["Ip"]), r["seed"], _params(c))
            out.append(tr.response(tr.image())[0].detach())
        return out
    if _tests(case) * (2 if kind in ("step", "denoised") else 1) > MAX_TESTS:
        return None
    d = _inputs(case, seed)
    if kind == "pose":  # the image and its loss at the pose; the adjoint's boundary terms have no 64-bit restatement here
        R, t = (np.asarray(a, np.float32) for a in pose_matrices())
        Rp = d["Rp"].astype(np.float64) @ R.T.astype(np.float64)
        d.update(verts=(d["verts"].astype(np.float64) @ R.T + t), Rp=Rp, tp=d["tp"] - Rp @ t)
    tr = _Tracer(case, d, seed, _params(case))
    Ec = tr.image()
    if kind == "render":
        return tr.response(Ec)[0].detach(), Ec
    target = _dev(d["target"]).to(_F)
    scale = 1.0 if case["loss"] == "l2" else 1.0 / target.numel()
    Ec.requires_grad_()
    Ic, cam = tr.response(Ec)
    img = Ic.detach()
    if kind == "denoised":
        guide = tr.guide()
        num, den = _gather(img, guide, case["radius"])
        img = num / den[..., None]
    diff = img - target
    loss = (0.5 * diff * diff).sum() if case["loss"] == "l2" else scale * diff.abs().sum()
    if kind == "pose":
        return Ic.detach(), loss, None
    dimg = diff if case["loss"] == "l2" else scale * diff.sign()
    if kind == "denoised":
        dimg = _gather(dimg / den[..., None], guide, case["radius"])[0]
    Ic.backward(dimg)
    dIp, dtex, dmat, dgp, dGp = tr.gradients(Ec.grad)
    if case["loss"] == "l2":
        return [Ic.detach(), loss, dIp]
    (la, ga), (lr, gr) = _tv(tr.alb, TV_WEIGHT), _tv(tr.rough, TV_WEIGHT)
    out = [Ic.detach(), loss, torch.stack([la, lr]), dtex[..., :3] + ga, dtex[..., 3] + gr,
           torch.cat([dgp, dGp.view(1), cam[0].grad, cam[1].grad.view(1), cam[2].grad])]
    return out + ([dmat[..., 0], dmat[..., 1:]] if case["principled"] else [])


def pose_matrices():
    """The rotation (Rodrigues) and translation of the pose case, from its pose parameters."""
    w, t = np.array([0.004, -0.003, 0.002]), np.array([0.003, -0.002, 0.004])
    th = float(np.linalg.norm(w))
    K = np.array([[0.0, -w[2], w[1]], [w[2], 0.0, -w[0]], [-w[1], w[0], 0.0]])
    return np.eye(3) + math.sin(th) / th * K + (1 - math.cos(th)) / th ** 2 * (K @ K), t
