"""Block shapes of the denoiser's levels on narrow, small and many images: each image of a stack is what the
oracle gives for it alone (the tolerance of the other denoiser tests)."""
import numpy as np
import pytest
import torch

from oracle import eawt as E
from tests.test_gpu_denoise import _inputs
from tests.test_gpu_parity import M, ctx  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,H,W,levels", [(1, 1, 1, 2), (70, 1, 1, 1), (130, 3, 2, 2), (9, 2, 5, 3), (5, 41, 7, 2),
                                          (300, 8, 8, 2), (3, 19, 9, 3), (2, 70, 24, 3), (2, 33, 33, 2), (1, 5, 40, 4),
                                          (2, 17, 36, 2), (3, 1, 65, 2), (2, 40, 96, 3), (1, 9, 130, 5)])
def test_every_block_shape(M, ctx, N, H, W, levels):  # noqa: F811
    kinds = [_inputs(M, ctx, 11 + i, H, W) for i in range(min(N, 3))]
    g = np.random.Generator(np.random.PCG64(N))
    pick = [int(k) for k in g.integers(0, len(kinds), N)]
    d3 = g.normal(size=(len(kinds), H, W, 3)).astype(np.float32)
    sig = (0.7, 0.5, 1.2)
    t = lambda a: torch.as_tensor(np.ascontiguousarray(a), device="cuda")  # noqa: E731
    img, nrm, pos = (t(np.stack([kinds[k][c] for k in pick])) for c in range(3))
    p = M.EawtParams(*sig, levels)
    rec = torch.empty(N * M.mirres_eawt_record_bytes(W, H, levels) // 4, device="cuda")
    out, gr = torch.full_like(img, -7.0), torch.full_like(img, -7.0)
    M.mirres_eawt_batch(ctx, img, nrm, pos, p, out, rec)
    M.mirres_eawt_batch_backward(ctx, t(d3[pick]), nrm, pos, p, rec, gr)
    torch.cuda.synchronize()
    out, gr = out.cpu().numpy(), gr.cpu().numpy()
    for k, (im, n, x) in enumerate(kinds):
        ref, orec = E.eawt(im, n, x, *sig, levels=levels)
        gref = E.eawt_backward(d3[k], orec)
        for i in [i for i in range(N) if pick[i] == k]:
            assert np.abs(out[i] - ref).max() <= 2e-5 * max(1.0, np.abs(ref).max())
            assert np.abs(gr[i] - gref).max() <= 2e-5 * max(1.0, np.abs(gref).max())
