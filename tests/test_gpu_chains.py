"""The default wavefront shape runs as two chains of half a wave: tape, images and history are those of
one chain, at totals around the sizes where a call is shared out."""
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


@pytest.mark.parametrize("sizes,reuse", [([(1, 1, 1)], 0), ([(256, 256, 1)], 0), ([(256, 257, 1)], 0),
                                         ([(401, 127, 3), (64, 33, 5)], 0), ([(300, 200, 2)] * 3, 4),
                                         ([(512, 300, 2), (31, 17, 3)], 4)])
def test_two_chains_equal_one(M, sizes, reuse):
    from paper_2406_16360_gb300.renderer import GpuWorkload
    views = []
    for k, (w, h, spp) in enumerate(sizes):
        K, c2w = synth.look_at((0.3 * k, 1.5, 4.0), (0.0, 1.0, 0.0), w, h, 40.0)
        views.append(synth.View(K, c2w, w, h, spp, 1 + k % 3, 0))
    out = []
    for one in (False, True):
        ctx = M.mirres_context_create(0)
        if one:
            M.mirres_set_wave_shape(ctx, M.mirres_get_wave_shape(ctx))  # set: one chain, as it is given
        gw = GpuWorkload(synth.Workload("chains", [synth.tiny_scene(subdiv=1)], views, ris_m=5), 0, ctx=ctx)
        tape, hist = torch.zeros_like(gw.new_tape()), gw.new_history() if reuse else None
        kw = dict(reuse=(reuse, 8), temporal=2, history=hist) if reuse else {}
        for seed in (3, 4):
            images, _ = gw.render(launch=1, tape=tape, seed=seed, **kw)
        torch.cuda.synchronize()
        out.append([tape] + images + ([hist] if reuse else []))
        for s in gw.scenes:
            s.close()
        ctx.close()
    assert all(torch.equal(a, b) for a, b in zip(*out))
