"""Gradient destinations shared by scenes of one adjoint call, above the size where the sums go through
packed accumulators: the shared arrays hold the sum of the scenes' own. d_images are positive, so that an
env texel's terms all are: FP32 sums of at most 2^21 such terms in another order differ by some
sqrt(2^21) 2^-24 = 9e-5 of the sum, within 1e-3 texel by texel; a lost addition misses a scene's share.
The other gradients have terms of either sign and keep 1e-3 of the tensor's largest."""
import numpy as np
import pytest
import torch

from paper_2406_16360_gb300 import synth
from tests.test_gpu_parity import M, ctx  # noqa: F401

pytestmark = pytest.mark.gpu
NAMES = ("albedo", "roughness", "metallic", "env", "verts")


@pytest.mark.parametrize("light", [0, 1])
@pytest.mark.parametrize("shared,same_handle", [(("env", "albedo"), False), (("env", "roughness", "metallic"), False),
                                                (NAMES, True)])
def test_shared_destinations_hold_the_sum(M, ctx, shared, same_handle, light):  # noqa: F811
    from paper_2406_16360_gb300.renderer import GpuWorkload
    scenes = [synth.object_scene(12 + s, 10, s, 24, 64, 32) for s in (0, 1)]
    views = []
    for k, (w, h, spp) in enumerate(((151, 97, 40), (131, 113, 40))):
        K, c2w = synth.look_at((3.2, 1.0, 1.0 + k), (0, 0, 0), w, h)
        views.append(synth.View(K, c2w, w, h, spp, 3, k))
    gw = GpuWorkload(synth.Workload("shared", scenes, views, ris_m=4, seed=3), 0, ctx=ctx)
    handles = [s.handle for s in gw.scenes]
    if same_handle:
        handles[1] = handles[0]
    assert gw.samples >= 1 << 20 and gw.samples >= sum(sum(t.numel() for t in s.params().values()) for s in gw.scenes)
    images, tape = gw.new_images(), gw.new_tape()
    M.mirres_render(ctx, handles, views, gw.params(1), images, tape)
    g = torch.Generator(device="cuda").manual_seed(1)
    d = [torch.rand(i.shape, device="cuda", generator=g) + 0.1 for i in images]
    call = M.mirres_light_backward if light else M.mirres_backward
    first = gw.scenes[0].params()
    own = [{k: torch.zeros_like(t) for k, t in (first if same_handle else s.params()).items()} for s in gw.scenes]
    call(ctx, handles, views, gw.params(1), d, tape, own)
    base = {k: own[0][k] * torch.rand(own[0][k].shape, device="cuda", generator=g) for k in shared}  # added to
    for rep in range(3):
        got = [{k: (base[k].clone() if k in shared else torch.zeros_like(t)) for k, t in o.items()} for o in own]
        for k in shared:
            got[1][k] = got[0][k]
        call(ctx, handles, views, gw.params(1), d, tape, got)
        torch.cuda.synchronize()
        for s in range(2):
            for k in NAMES:
                want = (own[0][k].double() + own[1][k].double() + base[k].double()) if k in shared else own[s][k].double()
                want = want.cpu().numpy()
                tol = dict(rtol=1e-3, atol=0) if k == "env" else dict(rtol=1e-3, atol=1e-3 * np.abs(want).max())
                np.testing.assert_allclose(got[s][k].cpu().numpy(), want, err_msg=k, **tol)
        assert all(float(o["env"].abs().max()) > 0 for o in own)
    for s in gw.scenes:
        s.close()
