"""The lane-refilling traversal kernels (leaves put aside while the warp goes on) against the
ray-by-ray traversal that the counting variant of the batched launch runs: same shading kernel,
so every tape word must be equal."""
import numpy as np
import pytest
import torch

from paper_2406_16360_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def M():
    import __graft_entry__
    __graft_entry__.build()
    from paper_2406_16360_gb300 import mirres
    return mirres


@pytest.fixture(scope="module")
def ctx(M):
    c = M.mirres_context_create(0)
    yield c
    c.close()


def _shells():
    """16 concentric spheres with holes: many leaves along every ray, paths that bounce between"""
    v, t = synth.icosphere(2)
    parts = []
    for k in range(16):
        keep = np.arange(len(t)) % 16 != k  # a different sixteenth of the faces missing in each
        parts.append((v * (0.4 + 0.05 * k), t[keep], synth.spherical_corner_uv(v, t[keep])))
    return synth.merge(parts)


def _funnel():
    """triangles shrinking by halves towards a corner: a tree far deeper than the shared stack"""
    tri = np.array([[0.0, 0.0, 0.0], [1.0, 0.1, 0.2], [0.2, 1.0, -0.1]])
    parts = [(np.array([-0.9, -0.9, -0.9]) + tri * 1.9 * 2.0 ** (-0.4 * k) + 0.9 * 2.0 ** (-0.4 * k),
              np.array([[0, 1, 2]]), np.array([[[0, 0], [1, 0], [0, 1]]], dtype=float)) for k in range(60)]
    return synth.merge(parts)


def _workload(mesh, width, height, spp, bounces):
    base = synth.tiny_scene()
    v, t, uv = {"shells": _shells, "funnel": _funnel, "one": lambda: (np.array([[-1, -1, 0], [1, -1, 0], [0, 1, 0]]),
                np.array([[0, 1, 2]]), np.array([[[0, 0], [1, 0], [0, 1]]], dtype=float))}[mesh]()
    sc = synth._scene(v, t, uv, base.albedo, base.roughness, base.metallic, base.env)
    K, c2w = synth.look_at((0.3, 0.4, 3.0), (0, 0, 0), width, height)
    return synth.Workload("trace", [sc], [synth.View(K, c2w, width, height, spp, bounces)], ris_m=4, seed=5)


@pytest.mark.parametrize("cap", [0, 25])
@pytest.mark.parametrize("mesh,width,height,spp,bounces", [("shells", 64, 48, 5, 5), ("shells", 1, 1, 1, 8),
                                                           ("shells", 33, 1, 1, 3), ("funnel", 61, 47, 3, 4),
                                                           ("one", 31, 3, 2, 3)])
def test_put_aside_leaves_change_nothing(M, ctx, mesh, width, height, spp, bounces, cap):
    """cap: an iteration limit of the caller's own, which rays must reach in both or neither"""
    from paper_2406_16360_gb300.renderer import GpuWorkload
    gw = GpuWorkload(_workload(mesh, width, height, spp, bounces), 0, ctx=ctx)
    tapes, images, capped = [], [], []
    for flags in (0, M.MIRRES_FLAG_COUNT_WORK):
        M.mirres_reset_counters(ctx)
        tape = torch.zeros_like(gw.new_tape())
        img, _ = gw.render(launch=1, tape=tape, flags=flags, max_visits=cap)
        torch.cuda.synchronize()
        out = (M.C.c_uint64 * 8)()
        M.lib().mirres_get_counters(ctx.handle, out)
        tapes.append(tape)
        images.append(img[0])
        capped.append(int(out[7]))
    M.mirres_reset_counters(ctx)
    assert torch.equal(tapes[0], tapes[1])
    assert torch.equal(images[0], images[1])
    assert capped[0] == capped[1] and (cap > 0 or capped[0] == 0)
    for s in gw.scenes:
        s.close()


@pytest.mark.parametrize("mesh", ["shells", "funnel", "one"])
@pytest.mark.parametrize("n", [1, 31, 33, 257, 400001])
def test_ray_queries_do_not_depend_on_their_neighbours(M, ctx, mesh, n):
    """lanes refilled from runs of 32 rays (400,001: more than one round of the grid): every ray's answer
    is the one it gets in another order, and any hit agrees with closest hit"""
    from paper_2406_16360_gb300.renderer import GpuWorkload
    gw = GpuWorkload(_workload(mesh, 8, 8, 1, 1), 0, ctx=ctx)
    h = gw.scenes[0].handle
    g = torch.Generator(device="cuda").manual_seed(n)
    o = torch.randn((n, 3), device="cuda", generator=g)
    d = 0.8 * torch.randn((n, 3), device="cuda", generator=g) - o
    rays = torch.cat([o, d / d.norm(dim=1, keepdim=True)], 1).contiguous()
    skip = torch.randint(-1, 3, (n,), device="cuda", generator=g, dtype=torch.int32)
    order = torch.randperm(n, device="cuda", generator=g)
    out = []
    for r, s in ((rays, skip), (rays[order].contiguous(), skip[order].contiguous())):
        tri, any_ = (torch.full((n,), -7, device="cuda", dtype=torch.int32) for _ in range(2))
        tuv = torch.full((n, 3), -7.0, device="cuda")
        M.mirres_trace(ctx, h, r, tri, tuv, skip=s)
        M.mirres_trace(ctx, h, r, any_, skip=s, any_hit=True)
        torch.cuda.synchronize()
        assert torch.equal(any_, torch.where(tri >= 0, 1, -1).to(torch.int32))
        out.append((tri, tuv))
    assert torch.equal(out[0][0][order], out[1][0]) and torch.equal(out[0][1][order], out[1][1])
    assert n < 31 or int((out[0][0] >= 0).sum()) > 0
    for s in gw.scenes:
        s.close()
