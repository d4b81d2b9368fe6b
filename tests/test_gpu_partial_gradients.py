"""Gradient destinations left out of an adjoint call above the size of the packed path: the others are
those of the whole call (same sums, another order of FP32 additions: 1e-3 of the tensor's largest, as in
the test of the packed path), and nothing is kept for the ones left out."""
import numpy as np
import pytest
import torch

from paper_2406_16360_gb300 import synth
from tests.test_gpu_parity import M, ctx  # noqa: F401

pytestmark = pytest.mark.gpu
NAMES = ("albedo", "roughness", "metallic", "env", "verts")
SUBSETS = [(), ("env",), ("albedo",), ("roughness",), ("metallic",), ("verts",), ("roughness", "metallic"),
           ("albedo", "verts"), ("env", "verts")]


def _workload(ctx, tex):  # noqa: F811
    from paper_2406_16360_gb300.renderer import GpuWorkload
    scenes = [synth.object_scene(12 + s, 10, s, tex + s, 64, 32) for s in (0, 1)]
    views = []
    for k, (w, h, spp) in enumerate(((211, 97, 60), (131, 157, 60))):
        K, c2w = synth.look_at((3.2, 1.0, 1.0 + k), (0, 0, 0), w, h)
        views.append(synth.View(K, c2w, w, h, spp, 2, k))
    return GpuWorkload(synth.Workload("partial", scenes, views, ris_m=4, seed=3), 0, ctx=ctx)


@pytest.mark.parametrize("light", [0, 1])
def test_subsets_equal_the_whole(M, ctx, light):  # noqa: F811
    gw = _workload(ctx, 24)
    assert gw.samples >= 1 << 20
    images, tape = gw.render(launch=1)
    d = [torch.randn(i.shape, device="cuda", generator=torch.Generator(device="cuda").manual_seed(1)) for i in images]
    call = M.mirres_light_backward if light else M.mirres_backward
    handles = [s.handle for s in gw.scenes]

    def grads(first, second):
        out = [{k: (torch.zeros_like(t) if k in names else None) for k, t in s.params().items()}
               for s, names in zip(gw.scenes, (first, second))]
        call(ctx, handles, gw.views, gw.params(1), d, tape, out)
        torch.cuda.synchronize()
        return out

    whole = grads(NAMES, NAMES)
    for i, names in enumerate(SUBSETS):
        got = grads(names, SUBSETS[(i + 4) % len(SUBSETS)])
        for s in range(2):
            for k in NAMES:
                if got[s][k] is not None:
                    want = whole[s][k].cpu().numpy()
                    np.testing.assert_allclose(got[s][k].cpu().numpy(), want, rtol=1e-3, atol=1e-3 * np.abs(want).max(),
                                               err_msg=f"{names} {k}")
    for s in gw.scenes:
        s.close()


def test_no_room_is_kept_for_destinations_left_out(M):  # noqa: F811
    """textures of 2 x 10^6 texels: the materials packed for reading are 32 bytes a texel, as many again
    would be their accumulators; a workspace grows by at most a quarter more than it needs, and 1 MB"""
    c = M.mirres_context_create(0)
    gw = _workload(c, 1000)
    texels = sum(s.roughness.numel() for s in gw.scenes)
    assert gw.samples >= sum(s.roughness.numel() + s.env.numel() // 3 + s.verts.shape[0] for s in gw.scenes)
    images, tape = gw.new_images(), gw.new_tape()
    gw.render(launch=2, images=images, tape=tape)  # the persistent launch keeps tables only
    out = [{k: (torch.zeros_like(t) if k == "env" else None) for k, t in s.params().items()} for s in gw.scenes]
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    gw.backward(images, tape, out, launch=2)
    torch.cuda.synchronize()
    used = before - torch.cuda.mem_get_info()[0]
    assert used <= 1.25 * 32 * texels + (8 << 20), (used, texels)
    assert all(float(o["env"].abs().max()) > 0 for o in out)
    gw.close()
