"""An adjoint whose packed accumulators find no room on the device: it runs without them, and the workspace
that the forward laid out stays where it is. 5000 x 5000 textures need 64 bytes a texel of packed scratch,
the workspace of a per-view launch holds 256 bytes for 2^22 samples; the device is filled (one allocation,
not touched) up to less than the difference."""
import numpy as np
import pytest
import torch

from paper_2406_16360_gb300 import synth

pytestmark = pytest.mark.gpu


def _workload(M, ctx, tex, size, spp):
    from paper_2406_16360_gb300.renderer import GpuWorkload
    s = synth.object_scene(12, 10, 0, 4, 64, 32)
    full = lambda *shape: torch.full(shape, 0.5, device="cuda")  # noqa: E731
    scene = synth.Scene(s.verts, s.tris, s.tri_uv, full(tex, tex, 3), full(tex, tex), full(tex, tex), s.env)
    K, c2w = synth.look_at((3.2, 1.0, 1.0), (0, 0, 0), size, size)
    return GpuWorkload(synth.Workload("limit", [scene], [synth.View(K, c2w, size, size, spp, 2, 0)], ris_m=2, seed=3), 0,
                       ctx=ctx)


def test_no_room_for_packed_accumulators():
    import __graft_entry__
    __graft_entry__.build()
    from paper_2406_16360_gb300 import mirres as M
    free = lambda: (torch.cuda.synchronize(), torch.cuda.mem_get_info()[0])[1]  # noqa: E731
    small = _workload(M, M.mirres_context_create(0), 16, 64, 1)  # loads the direct adjoint's kernels
    images, tape = small.render(launch=1)
    small.backward(images, tape, launch=1)
    small.close()
    gw = _workload(M, M.mirres_context_create(0), 5000, 640, 62)
    assert gw.samples >= 5000 * 5000 + 64 * 32 + gw.scenes[0].verts.shape[0]
    images, tape = gw.render(launch=0)
    want = gw.backward(images, tape, launch=0)[0]  # with room
    gw.close()
    gw = _workload(M, M.mirres_context_create(0), 5000, 640, 62)
    gw.render(launch=0, images=images, tape=tape)
    got = gw.zero_grads()
    torch.cuda.empty_cache()
    filler = torch.empty(free() - (200 << 20), dtype=torch.uint8, device="cuda")
    try:
        for _ in range(2):
            before = free()
            for t in got[0].values():
                t.zero_()
            gw.backward(images, tape, got, launch=0)
            assert before < 64 * 5000 * 5000
            assert abs(free() - before) <= 4 << 20
            gw.render(launch=0, images=images, tape=tape)
            assert abs(free() - before) <= 4 << 20
    finally:
        del filler
        torch.cuda.empty_cache()
    for k, t in got[0].items():
        a, b = t.cpu().numpy(), want[k].cpu().numpy()
        np.testing.assert_allclose(a, b, rtol=1e-3, atol=1e-3 * np.abs(b).max(), err_msg=k)
    gw.backward(images, tape, got, launch=0)  # with room again: added once more
    torch.cuda.synchronize()
    for k, t in got[0].items():
        b = 2 * want[k].cpu().numpy()
        np.testing.assert_allclose(t.cpu().numpy(), b, rtol=2e-3, atol=2e-3 * np.abs(b).max(), err_msg=k)
    gw.close()
