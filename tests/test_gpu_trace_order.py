"""Ray queries take three routes through the binary tree: one ray per thread up to a ray a lane, above that
bundles (rays of a camera in pixel order) one per thread and other orders by refilled lanes. A ray's answer
is the same on each, bit for bit."""
import numpy as np
import pytest
import torch

from paper_2406_16360_gb300 import synth
from tests.test_gpu_parity import M, ctx  # noqa: F401
from tests.test_gpu_trace_paths import _workload

pytestmark = pytest.mark.gpu


def _camera_rays(width, height):
    K, c2w = synth.look_at((0.3, 0.4, 3.0), (0, 0, 0), width, height)
    y, x = torch.meshgrid(torch.arange(height, device="cuda"), torch.arange(width, device="cuda"), indexing="ij")
    f = float(np.ravel(K)[0])
    d = torch.stack([(x + 0.5 - width / 2) / f, (y + 0.5 - height / 2) / f, torch.ones_like(x, dtype=torch.float32)], -1)
    R = torch.as_tensor(np.asarray(c2w, np.float32).reshape(3, 4), device="cuda")
    d = d.reshape(-1, 3) @ R[:, :3].T
    return torch.cat([R[:, 3].expand_as(d), d / d.norm(dim=1, keepdim=True)], 1).contiguous()


@pytest.mark.parametrize("mesh", ["shells", "funnel", "one"])
@pytest.mark.parametrize("width,height", [(487, 331), (401, 400), (640, 1601)])  # 161,197; 160,400; 1,024,640 rays
def test_every_route_gives_a_ray_the_same_answer(M, ctx, mesh, width, height):  # noqa: F811
    from paper_2406_16360_gb300.renderer import GpuWorkload
    gw = GpuWorkload(_workload(mesh, 8, 8, 1, 1), 0, ctx=ctx)
    h = gw.scenes[0].handle
    rays = _camera_rays(width, height)
    n = rays.shape[0]
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    assert n > 1024 * sms
    g = torch.Generator(device="cuda").manual_seed(n)
    skip = torch.randint(-1, 3, (n,), device="cuda", generator=g, dtype=torch.int32)

    def trace(r, s):
        tri, any_ = (torch.full((r.shape[0],), -7, device="cuda", dtype=torch.int32) for _ in range(2))
        tuv = torch.full((r.shape[0], 3), -7.0, device="cuda")
        M.mirres_trace(ctx, h, r, tri, tuv, skip=s)
        M.mirres_trace(ctx, h, r, any_, skip=s, any_hit=True)
        torch.cuda.synchronize()
        return tri, tuv, any_

    bundles = trace(rays, skip)
    order = torch.randperm(n, device="cuda", generator=g)
    mixed = trace(rays[order].contiguous(), skip[order].contiguous())
    parts = [trace(rays[i:i + 100003].contiguous(), skip[i:i + 100003].contiguous()) for i in range(0, n, 100003)]
    for k in range(3):
        assert torch.equal(bundles[k][order], mixed[k])
        assert torch.equal(bundles[k], torch.cat([p[k] for p in parts]))
    assert torch.equal(bundles[2], torch.where(bundles[0] >= 0, 1, -1).to(torch.int32))
    assert int((bundles[0] >= 0).sum()) > 0
    for s in gw.scenes:
        s.close()
