"""Tap weights of the denoiser are exact where the edge-stopping factors are one: with wide sigmas (every
exponent below 2^-60, and 2^x = 1 there) a level is the B3 convolution, and on whole numbers of eight bits
two levels of it need 24 bits: forward and adjoint are equal to the 64-bit convolution, bit for bit, away
from the image's edges (where k is not one)."""
import numpy as np
import pytest
import torch

from tests.test_gpu_parity import M, ctx  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,H,W,levels", [(1, 40, 70, 1), (2, 37, 131, 2), (3, 64, 33, 2), (1, 31, 29, 2)])
def test_wide_sigmas_give_the_exact_convolution(M, ctx, N, H, W, levels):  # noqa: F811
    g = np.random.Generator(np.random.PCG64(5))
    img, d = (g.integers(0, 256, (N, H, W, 3)).astype(np.float32) for _ in range(2))
    nrm, pos = (g.normal(size=(N, H, W, 3)).astype(np.float32) for _ in range(2))
    t = lambda a: torch.as_tensor(a, device="cuda")  # noqa: E731
    p = M.EawtParams(1e15, 1e15, 1e15, levels)
    rec = torch.empty(N * M.mirres_eawt_record_bytes(W, H, levels) // 4, device="cuda")
    out, gr = torch.empty_like(t(img)), torch.empty_like(t(img))
    M.mirres_eawt_batch(ctx, t(img), t(nrm), t(pos), p, out, rec)
    M.mirres_eawt_batch_backward(ctx, t(d), t(nrm), t(pos), p, rec, gr)
    torch.cuda.synchronize()
    margin = 2 * sum(2 * (1 << i) for i in range(levels))  # taps whose own k is one, in every level
    for src, got in ((img, out), (d, gr)):
        want = src.astype(np.float64)
        for i in range(levels):  # the filter is symmetric: the adjoint is the same convolution
            s = 1 << i
            for axis in (1, 2):
                want = sum(w * np.roll(want, (k - 2) * s, axis) for k, w in enumerate((1 / 16, 4 / 16, 6 / 16, 4 / 16, 1 / 16)))
        inner = (slice(None), slice(margin, H - margin), slice(margin, W - margin))
        assert want[inner].size > 0
        assert np.array_equal(got.cpu().numpy()[inner].astype(np.float64), want[inner])
