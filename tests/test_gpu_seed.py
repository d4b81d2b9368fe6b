"""A captured forward is replayed with another seed by rewriting its kernels' keys: every render equals
the one a fresh context makes with that seed."""
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


def _scene():
    return synth.tiny_scene(subdiv=1)


def _workload(n_views):
    views = []
    for k in range(n_views):
        K, c2w = synth.look_at((0.3 * k, 1.5, 4.0), (0.0, 1.0, 0.0), 160, 96, 40.0)
        views.append(synth.View(K, c2w, 160, 96, 5, 1 + k, 0))
    return synth.Workload("seed", [_scene()], views, ris_m=5)


def _render(gw, seed, reuse, grad_mode):
    kw = dict(reuse=(3, 4), temporal=2, history=gw.new_history()) if reuse else {}
    tape = torch.zeros_like(gw.new_tape(grad_mode))
    images, _ = gw.render(launch=1, tape=tape, seed=seed, grad_mode=grad_mode, **kw)
    torch.cuda.synchronize()
    return [tape] + [i.clone() for i in images]


@pytest.mark.parametrize("wave_log2,branches,reuse,grad_mode", [(25, 1, False, 0), (16, 1, False, 0), (16, 3, False, 1),
                                                                (16, 2, True, 0), (25, 1, True, 0)])
def test_seeds_replayed_equal_fresh_captures(M, wave_log2, branches, reuse, grad_mode):
    """one wave and many (over a chain or several), reservoir reuse, the FULL tape; seeds above 32 bits"""
    from paper_2406_16360_gb300.renderer import GpuWorkload

    def context():
        c = M.mirres_context_create(0)
        s = M.mirres_get_wave_shape(c)
        s.update(wave_log2=wave_log2, branches=branches)
        M.mirres_set_wave_shape(c, s)
        return c

    seeds = [0, 7, (5 << 32) | 7, 7, 0]
    kept = context()
    gw = GpuWorkload(_workload(3), 0, ctx=kept)
    got = []
    for s in seeds:  # one tape buffer, so that nothing but the seed changes between the calls
        if not got:
            tape, hist = gw.new_tape(grad_mode), gw.new_history() if reuse else None
        tape.zero_()
        kw = {}
        if reuse:
            hist.copy_(gw.new_history())
            kw = dict(reuse=(3, 4), temporal=2, history=hist)
        images, _ = gw.render(launch=1, tape=tape, seed=s, grad_mode=grad_mode, **kw)
        torch.cuda.synchronize()
        got.append([tape.clone()] + [i.clone() for i in images])
    for s in gw.scenes:
        s.close()
    for s, g in zip(seeds, got):
        fresh = context()
        gf = GpuWorkload(_workload(3), 0, ctx=fresh)
        want = _render(gf, s, reuse, grad_mode)
        assert all(torch.equal(a, b) for a, b in zip(g, want)), s
        for x in gf.scenes:
            x.close()
        fresh.close()
    assert not torch.equal(got[0][0], got[1][0]) and not torch.equal(got[1][0], got[2][0])
    kept.close()
