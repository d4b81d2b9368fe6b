"""Every primary ray of 2^21 samples escapes into one env texel: its gradient is the sum of d_image / spp
over the samples. Summed warp by warp in FP32 there are 2^21 / 32 additions, each off by at most half a
unit in the last place of the running sum, 2^-24 of it: at most 2^16 2^-24 = 2^-8 in all. Constant terms
round the same way again and again, so that 32 times as many additions drift well beyond that."""
import numpy as np
import pytest
import torch

from paper_2406_16360_gb300 import synth
from tests.test_gpu_parity import M, ctx  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("value", [1.0 / 3.0, 4.0 / 3.0])
def test_texel_of_all_escaping_rays(M, ctx, value):  # noqa: F811
    from paper_2406_16360_gb300.renderer import GpuWorkload
    scene = synth.object_scene(9, 8, 1, 5, 8, 4)
    th, ps = np.pi * 1.5 / 4, 2 * np.pi * 2.5 / 8 - np.pi  # a texel's centre
    away = np.array([np.sin(th) * np.sin(ps), np.cos(th), -np.sin(th) * np.cos(ps)])
    eye = 10.0 * away  # the object is behind the camera
    K, c2w = synth.look_at(eye, 2 * eye, 1024, 1024, 10.0)
    view = synth.View(K, c2w, 1024, 1024, 2, 1, 0)
    gw = GpuWorkload(synth.Workload("escape", [scene], [view], ris_m=1, seed=3), 0, ctx=ctx)
    images, tape = gw.render(launch=1)
    d = [torch.full_like(images[0], 2 * value)]
    env = gw.backward(d, tape, launch=1)[0]["env"].cpu().numpy().astype(np.float64)
    want = 2.0 ** 21 * float(np.float32(2 * value)) / 2
    hit = np.abs(env).sum(-1) > 0
    assert hit.sum() == 1
    np.testing.assert_allclose(env[hit][0], want, rtol=2.0 ** -8)
    for s in gw.scenes:
        s.close()
