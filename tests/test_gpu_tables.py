"""Hierarchy and environment tables at the edges of their kernels' tiles: blocks of 256 leaves,
radix tiles of 2048 keys scanned 256 at a time, rows and columns beyond one 1024-entry prefix
chunk, and guide tiles whose buckets fall on more texels than shared memory holds."""
import numpy as np
import pytest
import torch

from oracle import oracle as O
from oracle.material_smoothness import philox4x32_10
from paper_2406_16360_gb300 import synth
from tests.test_gpu_parity import M, _export_bvh, _mesh_scene, ctx  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [255, 256, 257, 511, 513, 2048, 2049, 530001])
def test_lbvh_at_tile_edges(M, ctx, n):  # noqa: F811
    from paper_2406_16360_gb300.renderer import DeviceScene
    rng = np.random.Generator(np.random.PCG64(n))
    v = (rng.normal(size=(n, 1, 3)) + 0.05 * rng.normal(size=(n, 3, 3))).reshape(-1, 3).astype(np.float32)
    sc = _mesh_scene(v, np.arange(3 * n).reshape(-1, 3))
    ds = DeviceScene(ctx, sc)
    for moved in (False, True):
        if moved:  # the same tree refitted to other vertices
            v2 = (v + rng.normal(scale=0.01, size=v.shape)).astype(np.float32)
            ds.verts.copy_(torch.as_tensor(v2, device="cuda"))
            M.mirres_bvh_refit(ds.handle)
        g = _export_bvh(M, ds, n)
        if not moved:
            o = O.lbvh(sc.verts, sc.tris)
            for k in ("keys", "left", "right", "parent", "lo", "hi"):
                assert np.array_equal(g[k], o[k]), k
        else:
            tri = v2.reshape(n, 3, 3)[(o["keys"] & np.uint64(0xFFFFFFFF)).astype(np.int64)]
            assert np.array_equal(g["lo"][n - 1:], tri.min(1)) and np.array_equal(g["hi"][n - 1:], tri.max(1))
            kid = lambda c: np.where(c >= 0, c, n - 1 + ~c)  # noqa: E731
            l, r = kid(g["left"]), kid(g["right"])
            assert np.array_equal(g["lo"][:n - 1], np.minimum(g["lo"][l], g["lo"][r]))
            assert np.array_equal(g["hi"][:n - 1], np.maximum(g["hi"][l], g["hi"][r]))
    ds.close()


@pytest.mark.parametrize("ew,eh,sun", [(1, 1, 1.0), (2051, 5, 1e3), (9, 2049, 1e3), (1024, 4, 1e9), (1025, 3, 1e-9)])
def test_env_tables_at_chunk_edges(M, ctx, ew, eh, sun):  # noqa: F811
    """thresholds against ordered FP64 sums, and a render whose draws go through the guide"""
    from paper_2406_16360_gb300.renderer import DeviceScene, GpuWorkload
    rng = np.random.Generator(np.random.PCG64(ew))
    sc = synth.tiny_scene(subdiv=1)
    sc.env = rng.uniform(0.1, 2.0, size=(eh, ew, 3)).astype(np.float32)
    sc.env[eh // 2, ew // 2] *= np.float32(sun)
    ds = DeviceScene(ctx, sc)
    flat = torch.zeros(eh * ew + 1, dtype=torch.int64, device="cuda")
    M.mirres_env_export_flat(ds.handle, flat)
    ref = O.OracleScene(sc).env_flat()
    got = flat.cpu().numpy().astype(np.float64) * 2.0 ** -53
    # the row's sine may differ by an ulp between the device and the host: a weight moves by 2^-52
    # of itself, a CDF value by a few such of its own size
    assert np.abs(got - ref).max() <= 2.0 ** -47
    assert np.all(np.diff(flat.cpu().numpy()) >= 0) and int(flat[-1]) == 2 ** 53
    # the draws of a render: the selected candidate's texel on the tape is the one its two random
    # words fall on (guide, then thresholds), found here by a search over all thresholds
    K, c2w = synth.look_at((0.0, 1.5, 4.0), (0.0, 1.0, 0.0), 64, 48, 40.0)
    w = synth.Workload("env", [sc], [synth.View(K, c2w, 64, 48, 4, 1)], ris_m=8, seed=2)
    gw = GpuWorkload(w, 0, ctx=ctx)
    _, tape = gw.render(launch=1)
    torch.cuda.synchronize()
    words = tape.cpu().numpy().reshape(-1, w.samples)
    cand, ytex = words[1], words[9]
    g = np.flatnonzero(cand >= 0)
    assert len(g)  # (few where the sun, below the horizon, draws nearly every candidate to itself)
    x = philox4x32_10(g // 4, g % 4, np.full_like(g, 1), cand[g], w.seed, 0)
    k = (x[0].astype(np.uint64) << np.uint64(21)) | (x[1].astype(np.uint64) >> np.uint64(11))
    want = np.searchsorted(flat.cpu().numpy().view(np.uint64), k, side="right") - 1
    assert np.array_equal(ytex[g], want)
    # and its direction that of the texel's row and column (FP32 angles: 1e-5)
    r, c = ytex[g] // ew, ytex[g] % ew
    th = np.pi * (r + ((x[3] & 0xFFFF) + 0.5) / 65536.0) / eh
    ps = 2.0 * np.pi * (c + ((x[3] >> 16) + 0.5) / 65536.0) / ew - np.pi
    want = np.stack([np.sin(th) * np.sin(ps), np.cos(th), -np.sin(th) * np.cos(ps)], 0)
    assert np.abs(words[10:13].view(np.float32)[:, g] - want).max() <= 1e-5
    for s in gw.scenes:
        s.close()
    ds.close()


@pytest.mark.parametrize("ew,eh", [(64, 32), (67, 33), (3, 1)])
def test_guide_over_black_texels(M, ctx, ew, eh):  # noqa: F811
    """rows and runs of black texels (equal thresholds, which a guide bucket may hold many of, or whose
    next entry lies far on): the draws of a render are those of a search over all thresholds"""
    from paper_2406_16360_gb300.renderer import GpuWorkload
    rng = np.random.Generator(np.random.PCG64(ew))
    sc = synth.tiny_scene(subdiv=1)
    sc.env = rng.uniform(0.1, 2.0, size=(eh, ew, 3)).astype(np.float32)
    sc.env[1:eh // 3] = 0.0
    sc.env[:, ew // 4:ew // 2] = 0.0
    sc.env[0, 0] = 1e-6  # a sliver of a bucket before the next threshold
    K, c2w = synth.look_at((0.0, 1.5, 4.0), (0.0, 1.0, 0.0), 64, 48, 40.0)
    w = synth.Workload("env", [sc], [synth.View(K, c2w, 64, 48, 4, 1)], ris_m=9, seed=2)
    gw = GpuWorkload(w, 0, ctx=ctx)
    flat = torch.zeros(eh * ew + 1, dtype=torch.int64, device="cuda")
    M.mirres_env_export_flat(gw.scenes[0].handle, flat)
    _, tape = gw.render(launch=1)
    torch.cuda.synchronize()
    words = tape.cpu().numpy().reshape(-1, w.samples)
    cand, ytex = words[1], words[9]
    g = np.flatnonzero(cand >= 0)
    assert len(g)
    x = philox4x32_10(g // 4, g % 4, np.full_like(g, 1), cand[g], w.seed, 0)
    k = (x[0].astype(np.uint64) << np.uint64(21)) | (x[1].astype(np.uint64) >> np.uint64(11))
    want = np.searchsorted(flat.cpu().numpy().view(np.uint64), k, side="right") - 1
    assert np.array_equal(ytex[g], want)
    for s in gw.scenes:
        s.close()
