"""The adjoint through packed materials and gradient accumulators (many samples per parameter)
against the one that reads and reduces into the caller's arrays directly (few): the same call with
one more scene, which no view uses and whose large textures move it across the line. Same terms,
another order of FP32 sums: up to 2^20 terms of either sign on one address keep 1e-3 of the tensor's
largest gradient."""
import numpy as np
import pytest
import torch

from paper_2406_16360_gb300 import synth
from tests.test_gpu_parity import M, ctx  # noqa: F401

pytestmark = pytest.mark.gpu
NAMES = ("albedo", "roughness", "metallic", "env", "verts")


def _scene(tex, ew, eh, seed):
    sc = synth.object_scene(9 + seed, 8, seed, tex, ew, eh)
    sc.env[:2] *= 0.05
    return sc


@pytest.mark.parametrize("normals", [0, 1])
@pytest.mark.parametrize("light", [0, 1])
@pytest.mark.parametrize("tex,ew,eh,full", [(1, 32, 16, 0), (5, 67, 33, 0), (48, 128, 64, 1)])
def test_packed_equals_direct(M, ctx, tex, ew, eh, full, light, normals):  # noqa: F811
    from paper_2406_16360_gb300.renderer import DeviceScene, GpuWorkload
    scenes = [_scene(tex, ew, eh, 1), _scene(tex + 2, ew, eh, 2)]
    views = []
    for k, (w, h, spp) in enumerate(((151, 97, 36), (131, 113, 36))):  # odd counts: warps across both scenes
        K, c2w = synth.look_at((3.2, 1.0, 1.0 + k), (0, 0, 0), w, h)
        views.append(synth.View(K, c2w, w, h, spp, 3, k))
    gw = GpuWorkload(synth.Workload("paths", scenes, views, ris_m=4, seed=3), 0, ctx=ctx, normals=normals)
    n_param = sum(s.albedo.numel() // 3 + s.env.numel() // 3 + s.verts.shape[0] for s in gw.scenes)
    assert gw.samples >= 1 << 20 and gw.samples >= n_param
    images, tape = gw.render(launch=1, grad_mode=full)
    g = torch.Generator(device="cuda").manual_seed(1)
    d = [torch.randn(i.shape, device="cuda", generator=g) for i in images]
    big = DeviceScene(ctx, synth.Scene(scenes[0].verts, scenes[0].tris, scenes[0].tri_uv, np.ones((1100, 1100, 3), np.float32),
                                       np.ones((1100, 1100), np.float32), np.ones((1100, 1100), np.float32), scenes[0].env))

    def grads(extra, skip=()):
        ds = gw.scenes + ([big] if extra else [])
        out = [{k: (None if k in skip else torch.zeros_like(t)) for k, t in s.params().items()} for s in ds]
        call = M.mirres_light_backward if light else M.mirres_backward
        call(ctx, [s.handle for s in ds], views, gw.params(1, grad_mode=full), d, tape, out)
        torch.cuda.synchronize()
        return out

    packed, direct, some = grads(False), grads(True), grads(False, skip=("albedo", "metallic", "verts"))
    assert all(not t.any() for t in direct[2].values())
    for s in range(2):
        for k in NAMES:
            a, b = packed[s][k].cpu().numpy(), direct[s][k].cpu().numpy()
            assert np.isfinite(a).all() and np.abs(b).max() > 0 or (k == "albedo" and light)
            np.testing.assert_allclose(a, b, rtol=1e-3, atol=1e-3 * np.abs(b).max(), err_msg=k)
            if some[s][k] is not None:
                np.testing.assert_allclose(some[s][k].cpu().numpy(), b, rtol=1e-3, atol=1e-3 * np.abs(b).max(), err_msg=k)
    for s in gw.scenes + [big]:
        s.close()
