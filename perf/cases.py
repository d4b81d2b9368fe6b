"""What the framework is timed on: calls as a program that uses it makes them.

Every case is one pass of such a program through the public entry points: a whole optimisation
step (render, image loss, adjoint), a render for viewing or serving, or one of the single calls
around them (hierarchy and environment tables, ray queries, denoiser, light regulariser). Sizes
are those of the repository's own workloads (`synth.config1` .. `config5`, the optimisation loop,
the denoiser and regulariser tests) or generic ones (odd image sizes, 1920 x 1080).

  listed()            the cases
  draw(rng)           one more of the same ranges
  prepare(case, seed) scenes, images and buffers on the GPU, made from the seed
  run(state)          one pass, returning all its outputs
  work(case)          bytes and operations a pass cannot do without
  exact(case, seed)   the outputs in 64 bits where plain torch gives them
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch
import torch.nn.functional as F

from paper_2406_16360_gb300 import mirres as M
from paper_2406_16360_gb300 import synth
from paper_2406_16360_gb300.renderer import GpuWorkload, MirresRender, scene_params

DEV = "cuda"
NAMES = ("albedo", "roughness", "metallic", "env", "verts")


# ----------------------------------------------------------------------------------------
# cases
# ----------------------------------------------------------------------------------------
def listed():
    return [
        # the smallest call: the tiny scene of config 1, forward and gradients, as an interactive
        # check or a unit test of a user's program makes it; launches and host time are all of it
        dict(name="preview-64", kind="step", mesh="tiny", lon=0, lat=0, tex=1, env_w=32, env_h=16, views=1, width=64,
             height=64, spp=4, bounces=2, ris=8, update="none", api="handle", full=0, reg=0),
        # one step of the optimisation loop on the 50k-triangle object of config 2 through the
        # autograd Function: env texels rewritten by the optimiser, a new random stream each step
        dict(name="optimise-50k", kind="step", mesh="object", lon=160, lat=157, tex=512, env_w=256, env_h=128, views=4,
             width=256, height=256, spp=8, bounces=3, ris=32, update="env", api="autograd", full=0, reg=0),
        # the multi-view batch of config 3 (499,036 triangles, 800 x 800, 16 spp, 4 bounces), 12
        # of its views: hierarchy and tables, forward, image loss, adjoint; the largest case
        dict(name="multiview-500k", kind="step", mesh="folds", lon=500, lat=500, tex=1024, env_w=1024, env_h=512,
             views=12, width=800, height=800, spp=16, bounces=4, ris=32, update="build", api="handle", full=0,
             reg=0),
        # geometry refinement: vertices moved, hierarchy refitted, odd image sizes, few
        # samples, mesh and material regularisers added to the gradients
        dict(name="geometry-120k", kind="step", mesh="object", lon=247, lat=243, tex=512, env_w=512, env_h=256, views=3,
             width=401, height=307, spp=4, bounces=2, ris=32, update="verts", api="handle", full=0, reg=1),
        # the adjoint through every vertex (grad_mode FULL) on a smaller object, odd sizes
        dict(name="full-adjoint-20k", kind="step", mesh="object", lon=101, lat=99, tex=256, env_w=256, env_h=128,
             views=3, width=317, height=203, spp=7, bounces=5, ris=32, update="none", api="handle", full=1,
             reg=0),
        # one finished picture: 1920 x 1080 at the paper's 32 samples per pixel, three bounces and
        # 512 x 256 env, forward only
        dict(name="still-1080p", kind="image", mesh="folds", lon=320, lat=313, tex=1024, env_w=512, env_h=256, views=1,
             width=1920, height=1080, spp=32, bounces=3, ris=32, reuse_k=0, reuse_r=0, temporal=0),
        # a frame of a sequence with spatial and temporal reservoir reuse (4 neighbours, radius 8)
        dict(name="reuse-frame-50k", kind="image", mesh="object", lon=160, lat=157, tex=512, env_w=256, env_h=128,
             views=2, width=400, height=304, spp=8, bounces=3, ris=32, reuse_k=4, reuse_r=8, temporal=2),
        # an uneven serving batch in the manner of config 5: scenes of 1k to 100k triangles, mixed
        # resolution, samples and bounces in one launch
        dict(name="serve-uneven-10", kind="serve", scenes=10, max_tris=100000, tex=256, env_w=256, env_h=128, ris=32,
             res=512, spp=16),
        # hierarchy and env tables alone for config 3's mesh and env (topology or meshing changed)
        dict(name="rebuild-500k", kind="build", mesh="folds", lon=500, lat=500, env_w=1024, env_h=512),
        # visibility queries of another program: a million rays, closest hit and any hit
        dict(name="rays-1m", kind="rays", mesh="object", lon=160, lat=157, n=1048579, any=0, both=1),
        # the denoiser and its adjoint between the rendered views and the loss, a stack of 8
        dict(name="denoise-8x800", kind="denoise", views=8, width=800, height=800, levels=3),
        # the monochrome light regulariser on a rendered batch: lighting, loss, adjoint
        dict(name="light-50k", kind="light", mesh="object", lon=160, lat=157, tex=512, env_w=256, env_h=128, views=4,
             width=256, height=256, spp=8, bounces=3, ris=32),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _object(rng, lo=2000, hi=500000):
    n = max(8, int(math.sqrt(_log(rng, lo, hi) / 2)))
    return dict(mesh=rng.choice(["object", "folds"]), lon=n + rng.randrange(0, 4), lat=n - rng.randrange(0, 4))


def _env(rng):
    h = rng.choice([16, 64, 100, 128, 256, 512])
    return dict(env_w=2 * h, env_h=h)


def draw(rng: random.Random):
    kind = rng.choice(["step", "step", "step", "image", "image", "serve", "build", "rays", "denoise", "light"])
    if kind == "denoise":
        w, h = _log(rng, 33, 1000), _log(rng, 33, 1000)
        return dict(kind=kind, views=rng.randrange(1, 9), width=w, height=h, levels=rng.randrange(1, 6))
    if kind == "build":
        return dict(kind=kind, **_object(rng), **_env(rng))
    if kind == "rays":
        return dict(kind=kind, **_object(rng), n=_log(rng, 1000, 1 << 20), any=rng.randrange(2), both=0)
    if kind == "serve":
        return dict(kind=kind, scenes=rng.randrange(2, 11), max_tris=_log(rng, 5000, 100000), tex=rng.choice([64, 256]),
                    env_w=256, env_h=128, ris=rng.choice([16, 32]), res=rng.choice([128, 256, 512]),
                    spp=rng.choice([4, 8, 16]))
    w, h = _log(rng, 61, 700), _log(rng, 61, 700)
    spp = rng.choice([1, 3, 4, 8, 16, 32])
    most = 30_000_000 if kind != "image" else 60_000_000  # samples, below the largest listed case
    views = max(1, min(_log(rng, 1, 16), most // (w * h * spp)))
    c = dict(kind=kind, **_object(rng), tex=rng.choice([128, 256, 512, 1000]), **_env(rng), views=views, width=w,
             height=h, spp=spp, bounces=rng.randrange(1, 6), ris=rng.choice([8, 16, 32, 33]))
    if kind == "step":
        full = rng.random() < 0.25
        c.update(update=rng.choice(["none", "env", "verts", "build"]), api=rng.choice(["handle", "autograd"]),
                 full=int(full), reg=int(rng.random() < 0.3))
        if full:
            c["api"] = "handle"  # the autograd Function has the PRIMARY adjoint only
        if c["api"] == "autograd":
            c["reg"] = 0
    elif kind == "image":
        reuse = rng.random() < 0.3
        c.update(reuse_k=rng.randrange(1, 6) if reuse else 0, reuse_r=rng.randrange(2, 17) if reuse else 0,
                 temporal=rng.choice([0, 2]) if reuse else 0)
    return c


# ----------------------------------------------------------------------------------------
# inputs
# ----------------------------------------------------------------------------------------
def _gen(seed, salt=0):
    g = torch.Generator(device=DEV)
    g.manual_seed((seed * 1_000_003 + salt) & 0x7FFFFFFFFFFF)
    return g


def _texture(n, channels, g, lo=0.05, hi=0.95):
    """smooth noise in [lo, hi]: three octaves of random lattices, bilinear"""
    out = torch.zeros((1, channels, n, n), device=DEV)
    amp, norm = 1.0, 0.0
    for lattice in (9, 17, 33):
        r = torch.rand((1, channels, lattice, lattice), device=DEV, generator=g) * 2 - 1
        out += amp * F.interpolate(r, size=(n, n), mode="bilinear", align_corners=True)
        norm += amp
        amp *= 0.5
    t = (lo + (hi - lo) * (0.5 + 0.5 * out / norm))[0]
    return t.permute(1, 2, 0).contiguous()


def _environment(w, h, g):
    """log-normal texels and a 2 x 2 sun in the upper half, as synth.env_lognormal_sun"""
    env = torch.exp(1.5 * torch.randn((h, w, 3), device=DEV, generator=g))
    r = int(torch.randint(h // 8, max(h // 3, h // 8 + 1), (1,), device=DEV, generator=g))
    c = int(torch.randint(0, w - 2, (1,), device=DEV, generator=g))
    env[r:r + 2, c:c + 2, :] = 1e3
    return env


def _mesh(case, seed):
    if case["mesh"] == "tiny":
        s = synth.tiny_scene()
        return s.verts, s.tris, s.tri_uv
    folds = 0.1 if case["mesh"] == "folds" else 0.0
    v, t, uv = synth.merge([synth.displaced_sphere(case["lon"], case["lat"], seed % 100003, 0.15, folds)]
                           + synth.occluder_boxes(seed % 100003))
    return v.astype(np.float32), t.astype(np.int32), uv.astype(np.float32)


def _scene(case, seed):
    g = _gen(seed, 1)
    v, t, uv = _mesh(case, seed)
    n = case.get("tex", 4)
    if case["mesh"] == "tiny":
        env = torch.full((case["env_h"], case["env_w"], 3), 0.2, device=DEV)
        env[3, seed % case["env_w"], :] = 500.0
        alb, rough, metal = (torch.full(s, x, device=DEV) for s, x in (((1, 1, 3), 0.5), ((1, 1), 0.5), ((1, 1), 0.0)))
    else:
        env = _environment(case["env_w"], case["env_h"], g) if "env_w" in case else torch.ones((16, 32, 3), device=DEV)
        alb = _texture(n, 3, g)
        rough, metal = _texture(n, 1, g)[..., 0].contiguous(), _texture(n, 1, g)[..., 0].contiguous()
    return synth.Scene(v, t, uv, alb, rough, metal, env)


def _cameras(n, w, h, spp, bounces, seed):
    rng = np.random.Generator(np.random.PCG64(seed + 555))
    views = []
    for _ in range(n):
        a, el = rng.uniform(0, 2 * np.pi), np.arcsin(rng.uniform(math.sin(math.radians(8)), math.sin(math.radians(75))))
        eye = 3.5 * np.array([math.cos(el) * math.cos(a), math.sin(el), math.cos(el) * math.sin(a)])
        K, c2w = synth.look_at(eye, (0, 0, 0), w, h)
        views.append(synth.View(K, c2w, w, h, spp, bounces, 0))
    return views


class Program:
    """What a user's program keeps: a workload on the GPU, its buffers and the step number."""

    def __init__(self, case, seed):
        self.case, self.seed, self.step, self.gw = case, seed, 0, None

    def close(self):
        if self.gw is not None:
            gw, self.gw = self.gw, None
            gw.close()

    def __del__(self):
        self.close()


def _workload(case, seed):
    if case["mesh"] == "tiny":
        K, c2w = synth.look_at((0.0, 1.5, 4.0), (0.0, 1.0, 0.0), case["width"], case["height"], 40.0)
        views = [synth.View(K, c2w, case["width"], case["height"], case["spp"], case["bounces"])]
    else:
        views = _cameras(case["views"], case["width"], case["height"], case["spp"], case["bounces"], seed)
    w = synth.Workload("perf", [_scene(case, seed)], views, case["ris"], seed=seed)
    return GpuWorkload(w, 0)


def prepare(case, seed):
    st = Program(case, seed)
    kind = case["kind"]
    g = _gen(seed, 2)
    if kind == "denoise":
        st.ctx = M.mirres_context_create(0)
        st.image, st.normal, st.position, st.d_out = _denoise_inputs(case, g)
        st.params = M.EawtParams(0.5, 0.3, 0.2, case["levels"])
        n = case["views"] * M.mirres_eawt_record_bytes(case["width"], case["height"], case["levels"])
        st.record = torch.empty(n // 4, device=DEV, dtype=torch.float32)
        st.out, st.d_image = torch.empty_like(st.image), torch.empty_like(st.image)
        st.gw = st.ctx  # closed with the program
    elif kind == "serve":
        rng = np.random.Generator(np.random.PCG64(seed + 2024))
        scenes, views = [], []
        for s in range(case["scenes"]):
            # the sizes are the case's, not the seed's: log-uniform over the range
            q = (s + 0.5) / case["scenes"]
            n = max(4, int(math.sqrt(1000.0 * (case["max_tris"] / 1000.0) ** q / 2.0)))
            scenes.append(_scene(dict(case, mesh="object", lon=n, lat=n), seed + 31 * s))
            res = max(64, case["res"] >> ((3 * s + 1) % 3))
            a = rng.uniform(0, 2 * np.pi)
            K, c2w = synth.look_at((3.5 * math.cos(a), 1.0, 3.5 * math.sin(a)), (0, 0, 0), res, res)
            views.append(synth.View(K, c2w, res, res, max(1, case["spp"] >> (s % 3)), 2 + s % 4, s))
        st.gw = GpuWorkload(synth.Workload("perf", scenes, views, case["ris"], seed=seed), 0)
        st.images, st.tape = st.gw.new_images(), st.gw.new_tape()
    elif kind in ("build", "rays"):
        c = dict(case, width=16, height=16, spp=1, bounces=1, ris=1, views=1)
        st.gw = _workload(c, seed)
        if kind == "build":
            Fn, H, W = st.gw.scenes[0].tris.shape[0], case["env_h"], case["env_w"]
            i32, f32 = dict(device=DEV, dtype=torch.int32), dict(device=DEV, dtype=torch.float32)
            st.tree = dict(keys=torch.empty(Fn, device=DEV, dtype=torch.int64), left=torch.empty(Fn - 1, **i32),
                           right=torch.empty(Fn - 1, **i32), parent=torch.empty(2 * Fn - 1, **i32),
                           lo=torch.empty((2 * Fn - 1, 3), **f32), hi=torch.empty((2 * Fn - 1, 3), **f32))
            st.env = dict(marg=torch.empty(H + 1, **i32), cond=torch.empty((H, W + 1), **i32),
                          texel=torch.empty((H, W, 4), **f32), total=torch.empty(1, device=DEV, dtype=torch.float64))
            st.flat = torch.empty(H * W + 1, device=DEV, dtype=torch.int64)
        else:
            n = case["n"]
            o = torch.randn((n, 3), device=DEV, generator=g)
            out = torch.arange(n, device=DEV)[:, None] % 2 == 0  # cameras outside, points near the surface
            o = torch.where(out, 3.5 * o / o.norm(dim=1, keepdim=True),
                            (1.0 + torch.rand((n, 1), device=DEV, generator=g)) * o / o.norm(dim=1, keepdim=True))
            d = torch.randn((n, 3), device=DEV, generator=g)
            d = torch.where(out, 1.2 * d / d.norm(dim=1, keepdim=True) - o, d)
            st.rays = torch.cat([o, d / d.norm(dim=1, keepdim=True)], 1).contiguous()
            st.hits = [torch.empty(n, device=DEV, dtype=torch.int32) for _ in range(2)]
            st.tuv = torch.empty((n, 3), device=DEV)
    else:
        st.gw = _workload(case, seed)
        gw, sc = st.gw, st.gw.scenes[0]
        st.images, st.refs = gw.new_images(), [torch.rand((v.height, v.width, 3), device=DEV, generator=g) for v in gw.views]
        if kind == "step":
            st.env = sc.env.clone()
            st.verts = sc.verts * (1 + 1e-3 * torch.randn(sc.verts.shape, device=DEV, generator=g))
            st.rest = sc.verts.clone()
            if case["api"] == "autograd":
                st.refs = torch.stack(st.refs)
                for p in scene_params(gw):
                    p.requires_grad_(True)
            else:
                st.tape, st.grads = gw.new_tape(case["full"]), gw.zero_grads()
                st.d = [torch.empty_like(i) for i in st.images]
                st.loss = torch.zeros(1, device=DEV)
                st.lk = M.LkParams(0.02, 1e3, 1e3, seed & 0xFFFFFFFF, 0, 0.0)
        elif kind == "image":
            st.tape = gw.new_tape()
            st.history = gw.new_history() if case["temporal"] else None
        else:  # light: the tape of a render is what its calls start from
            st.images, st.tape = gw.render(launch=1, images=st.images)
            st.demod = [torch.empty((v.height, v.width, 4), device=DEV) for v in gw.views]
            st.grads, st.loss = gw.zero_grads(), torch.zeros(1, device=DEV)
    return st


# ----------------------------------------------------------------------------------------
# one pass
# ----------------------------------------------------------------------------------------
def _update(st):
    """what the optimiser rewrote since the last step"""
    sc, how = st.gw.scenes[0], st.case["update"]
    with torch.no_grad():
        if how in ("env", "verts"):
            sc.env.copy_(st.env)
        if how == "verts":
            sc.verts.copy_(st.verts)
    if how == "build":
        M.mirres_bvh_build(sc.handle)


def _step(st):
    gw, case = st.gw, st.case
    seed = st.seed + st.step  # a new random stream each step
    st.step += 1
    _update(st)
    if case["api"] == "autograd":
        params = scene_params(gw)
        for p in params:
            p.grad = None
        img = MirresRender.apply(gw, 1, seed, *params)
        loss = ((img - st.refs) ** 2).sum()
        loss.backward()
        return dict(images=img.detach(), loss=loss.detach(), **{n: p.grad for n, p in zip(NAMES, params)})
    full = case["full"]
    gw.render(launch=1, images=st.images, tape=st.tape, seed=seed, grad_mode=full)
    st.loss.zero_()
    for i, r, d in zip(st.images, st.refs, st.d):
        M.mirres_l2_loss(i, r, d, st.loss)
    for t in st.grads[0].values():
        t.zero_()
    gw.backward(st.d, st.tape, st.grads, launch=1, seed=seed, grad_mode=full)
    g = st.grads[0]
    if case["reg"]:
        h = gw.scenes[0].handle
        M.mirres_mesh_regularizers(gw.ctx, h, st.rest, 10.0, 1.0, st.loss, g["verts"])
        M.mirres_material_smoothness(gw.ctx, h, gw.views[0], 0, st.lk, st.loss, g["albedo"], g["roughness"], g["verts"])
    return dict(images=st.images, loss=st.loss, **g)


def run(st):
    case, kind = st.case, st.case["kind"]
    if kind == "step":
        return _step(st)
    if kind == "image":
        st.gw.render(launch=1, images=st.images, tape=st.tape, reuse=(case["reuse_k"], case["reuse_r"]),
                     temporal=case["temporal"], history=st.history)
        if st.history is None:
            return st.images
        n = st.history.numel() // 5
        return dict(images=st.images, selection=st.history[:2 * n], weights=st.history[2 * n:].view(torch.float32))
    if kind == "serve":
        st.gw.render(launch=1, images=st.images, tape=st.tape)
        return st.images
    if kind == "build":
        h = st.gw.scenes[0].handle
        M.mirres_bvh_build(h)
        M.mirres_bvh_export(h, **st.tree)
        M.mirres_env_export(h, **st.env)
        M.mirres_env_export_flat(h, st.flat)
        return dict(**st.tree, **st.env, flat=st.flat)
    if kind == "rays":
        h = st.gw.scenes[0].handle
        out = {}
        if case["both"] or not case["any"]:
            M.mirres_trace(st.gw.ctx, h, st.rays, st.hits[0], st.tuv)
            out.update(tri=st.hits[0], tuv=st.tuv)
        if case["both"] or case["any"]:
            M.mirres_trace(st.gw.ctx, h, st.rays, st.hits[1], any_hit=True)
            out.update(any=st.hits[1])
        return out
    if kind == "denoise":
        M.mirres_eawt_batch(st.ctx, st.image, st.normal, st.position, st.params, st.out, st.record)
        M.mirres_eawt_batch_backward(st.ctx, st.d_out, st.normal, st.position, st.params, st.record, st.d_image)
        return dict(out=st.out, d_image=st.d_image)
    st.loss.zero_()
    for t in st.grads[0].values():
        t.zero_()
    st.gw.light_demod(st.tape, launch=1, demod=st.demod)
    _, d = st.gw.light_loss(st.demod, st.refs, 1e3, st.loss)
    st.gw.light_backward(d, st.tape, st.grads, launch=1)
    return dict(demod=st.demod, loss=st.loss, d_demod=d, **st.grads[0])


# ----------------------------------------------------------------------------------------
# what a pass cannot do without
# ----------------------------------------------------------------------------------------
def work(case):
    kind = case["kind"]
    if kind == "denoise":
        n = case["views"] * case["width"] * case["height"]
        # image, normal, position, d_out in; out and d_image out; 25 taps with three squared
        # differences, an exponential and four sums, per level and direction
        return dict(bytes=n * 3 * 4 * 6, flops=n * case["levels"] * 2 * 25 * 32)
    if kind == "serve":
        out = dict(bytes=0.0, flops=0.0)
        for s in range(case["scenes"]):
            q = (s + 0.5) / case["scenes"]
            f = 1000.0 * (case["max_tris"] / 1000.0) ** q
            res = max(64, case["res"] >> ((3 * s + 1) % 3))
            w = _render_work(f, case["tex"], case["env_w"] * case["env_h"], res * res, max(1, case["spp"] >> (s % 3)),
                             2 + s % 4, case["ris"])
            out = {k: out[k] + w[k] for k in out}
        return out
    tris = 1282 if case["mesh"] == "tiny" else 2 * case["lon"] * (case["lat"] - 1) + 36
    texels = case.get("env_w", 32) * case.get("env_h", 16)
    if kind == "build":  # vertices and indices in; tree, boxes and env tables out
        return dict(bytes=tris * (6 + 12 + 8 + 16 + 48) + texels * (12 + 16 + 4 + 8), flops=tris * 60 + texels * 20)
    if kind == "rays":
        passes = 2 if case["both"] else 1
        return dict(bytes=passes * case["n"] * (24 + 10) + tris * 64,
                    flops=passes * case["n"] * (24 * math.log2(tris) + 54))
    pix = case["views"] * case["width"] * case["height"]
    w = _render_work(tris, case["tex"], texels, pix, case["spp"], case["bounces"], case["ris"])
    params = case["tex"] ** 2 * 20 + texels * 12 + tris * 6
    if kind == "light":  # the tape's words of the primary vertices in, lighting and gradients out
        n = pix * case["spp"]
        return dict(bytes=n * 68 + pix * (16 + 12 + 12) + 2 * params, flops=n * 600)
    if kind == "step":  # plus reference images, image gradients and the parameters' gradients
        w["bytes"] += pix * 24 + params
        w["flops"] += pix * case["spp"] * 500 * (case["bounces"] if case["full"] else 1)
    return w


def _render_work(tris, tex, texels, pix, spp, bounces, ris):
    """scene read once, image written once; about 0.7 of the paths go on to each further bounce,
    a vertex takes `ris` candidates of 80 operations, a ray two box tests a level and a triangle"""
    rays = sum(0.7 ** b * (1 if b else 1) for b in range(bounces)) * 1.7
    verts = sum(0.7 ** (b + 1) for b in range(bounces))
    n = pix * spp
    return dict(bytes=tris * (6 + 12 + 24) + tex * tex * 20 + texels * 12 + pix * 12,
                flops=n * (verts * ris * 80 + rays * (24 * math.log2(max(tris, 2)) + 54)))


# ----------------------------------------------------------------------------------------
# outputs in 64 bits
# ----------------------------------------------------------------------------------------
def _denoise_inputs(case, g):
    """noisy HDR images of a round object before a distant background, its normals and positions"""
    N, H, W = case["views"], case["height"], case["width"]
    y, x = torch.meshgrid(torch.linspace(-1, 1, H, device=DEV), torch.linspace(-1, 1, W, device=DEV), indexing="ij")
    r2 = (x * x + y * y)[None].expand(N, H, W) / (0.3 + 0.5 * torch.rand((N, 1, 1), device=DEV, generator=g))
    inside = (r2 < 1)[..., None]
    z = torch.sqrt((1 - r2).clamp_min(0))
    n = torch.stack([x.expand(N, H, W), y.expand(N, H, W), z], -1)
    n = n + 0.05 * torch.randn(n.shape, device=DEV, generator=g)
    n = torch.where(inside, n / n.norm(dim=-1, keepdim=True), torch.zeros_like(n)).contiguous()
    p = torch.where(inside, torch.stack([x.expand(N, H, W), y.expand(N, H, W), z], -1), torch.zeros_like(n)).contiguous()
    img = torch.exp(0.6 * torch.randn((N, H, W, 3), device=DEV, generator=g)) * (0.3 + 0.7 * z[..., None])
    return img.contiguous(), n, p, torch.randn((N, H, W, 3), device=DEV, generator=g)


def _taps(step, H, W):
    b3 = (1 / 16, 4 / 16, 6 / 16, 4 / 16, 1 / 16)
    for a in range(5):
        for b in range(5):
            dy, dx = (a - 2) * step, (b - 2) * step
            if abs(dy) >= H or abs(dx) >= W:
                continue
            yp, yq = slice(max(0, -dy), H - max(0, dy)), slice(max(0, dy), H - max(0, -dy))
            xp, xq = slice(max(0, -dx), W - max(0, dx)), slice(max(0, dx), W - max(0, -dx))
            yield b3[a] * b3[b], (yp, xp), (yq, xq)


def exact(case, seed):
    kind = case["kind"]
    g = _gen(seed, 2)
    if kind == "denoise":
        image, normal, position, d_out = (t.double() for t in _denoise_inputs(case, g))
        H, W = case["height"], case["width"]
        sn, sx = float(np.float32(0.3)), float(np.float32(0.2))
        out, d_image = torch.empty_like(image), torch.empty_like(image)
        for v in range(case["views"]):
            c, nv, pv, levels = image[v], normal[v], position[v], []
            weights = lambda c, h, p, q, s: h * torch.exp(  # noqa: E731
                -((c[p] - c[q]) ** 2).sum(-1) / s ** 2 - ((nv[p] - nv[q]) ** 2).sum(-1) / sn ** 2
                - ((pv[p] - pv[q]) ** 2).sum(-1) / sx ** 2)
            for i in range(case["levels"]):
                s = 0.5 / 2 ** i
                acc, k = torch.zeros_like(c), torch.zeros((H, W), device=DEV, dtype=torch.float64)
                for h, p, q in _taps(1 << i, H, W):
                    w = weights(c, h, p, q, s)
                    acc[p] += w[..., None] * c[q]
                    k[p] += w
                levels.append((c, k, s))
                c = acc / k[..., None]
            out[v] = c
            d = d_out[v]
            for i in reversed(range(case["levels"])):
                c, k, s = levels[i]
                gk, acc = d / k[..., None], torch.zeros_like(d)
                for h, p, q in _taps(1 << i, H, W):
                    acc[p] += weights(c, h, p, q, s)[..., None] * gk[q]
                d = acc
            d_image[v] = d
        return dict(out=out, d_image=d_image)
    if kind == "build":  # the env tables' probabilities; the tree's boxes depend on its topology
        env = _environment(case["env_w"], case["env_h"], _gen(seed, 1)).double()
        H, W = case["env_h"], case["env_w"]
        st = torch.sin(math.pi * (torch.arange(H, device=DEV, dtype=torch.float64) + 0.5) / H)
        w = env.mean(-1) * st[:, None]
        total = w.sum()
        return dict(texel=torch.cat([env, (w / total * (H * W))[..., None]], -1), total=total.reshape(1))
    # renders: every sample follows discrete decisions of single-precision arithmetic (which
    # candidate, which triangle), so a 64-bit evaluation has other paths and no value to compare
    return None
