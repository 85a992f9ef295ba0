"""Image traces cull whole 8x4-pixel tiles before the trace.  Every form the
tile bound must accept or step aside for -- part counts around its limits,
ragged images, rays with origins of their own, rays no cone bounds, entries
that are not rays -- gives the hits and flags of the trace without tiles bit
for bit."""

from __future__ import annotations

import numpy as np
import pytest

import synthetic

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__

    __graft_entry__.build()
    import paper_1911_06001_gb300 as g

    c = g.Context(0)
    yield c
    c.check_device()
    c.close()


@pytest.fixture(scope="module")
def pool(ctx):
    p = synthetic.asset_pool(range(6, 8), 2, seed=3)
    return p, [ctx.upload(a.asset.depth, a.asset.leaf_ids, a.asset.rgb) for a in p]


def _scene(ctx, pool, parts, seed):
    bat = synthetic.batched_scenes(seed=seed, n_scenes=1, parts=(parts, parts), depths=range(6, 8), side=(8, 9),
                                   per_depth=2, pool=pool[0])
    s = bat.scenes[0]
    sc = ctx.scene([pool[1][int(a)] for a in s.part_asset], s.parent)
    sc.set_transforms(s.local)
    sc.refit()
    return sc, s


def _rays(kind, w, h, box, seed):
    rng = np.random.default_rng(seed)
    if kind == "incoherent":
        return synthetic.random_rays(w * h, rng, (-box / 2,) * 3, (box / 2,) * 3)
    eye = np.array([0.1, 0.2, 1.0]) * (box if kind != "close" else 0.3 * box)
    r = synthetic.pinhole_rays(eye, (0.0, 0.0, 0.0), w, h, 60.0 if kind != "wide" else 150.0)
    if kind == "lens":  # origins spread over a lens, directions of any length, bounded segments
        r[:, :3] += (0.05 * rng.standard_normal((w * h, 3))).astype(np.float32)
        r[:, 4:7] *= rng.uniform(0.1, 10.0, (w * h, 1)).astype(np.float32)
        r[:, 7] = np.where(rng.random(w * h) < 0.5, np.inf, box)
    if kind == "broken":  # entries that are not rays, and rays that reach behind their origin
        r[::7, 4:7] = 0.0
        r[3::11, 0] = np.nan
        r[5::13, 3], r[5::13, 7] = 2.0, 1.0
        r[w * h // 2::3, 3] = -box
        r[:32 * (w // 8), 4:7] = np.nan
    return r.astype(np.float32)


def _trace(sc, rays, flags, hits=None):
    import torch

    r = torch.from_numpy(np.ascontiguousarray(rays)).cuda()
    rf = torch.full((r.shape[0],), 77, dtype=torch.int32, device="cuda")
    h = sc.trace(r, hits=hits, flags=flags, ray_flags=rf)
    torch.cuda.synchronize()
    return h.cpu().numpy(), rf.cpu().numpy()


@pytest.mark.parametrize("kind", ["pinhole", "close", "wide", "lens", "broken", "incoherent"])
@pytest.mark.parametrize("parts", [8, 20, 31, 32, 33, 63, 64, 65, 200])
def test_tiles_do_not_change_results(ctx, pool, parts, kind):
    import paper_1911_06001_gb300 as g

    sc, s = _scene(ctx, pool, parts, 100 + parts)
    w, h = (263, 131) if parts % 2 else (256, 128)  # 33 x 33 tiles with ragged edges, 32 x 32 whole ones
    rays = _rays(kind, w, h, s.meta["box"], parts)
    ref = _trace(sc, rays, g.TRACE_DEFAULT)
    for extra in (0, g.TRACE_GRID):
        got = _trace(sc, rays, g.TRACE_DEFAULT | g.trace_image(w) | extra)
        assert np.array_equal(got[0], ref[0]) and np.array_equal(got[1], ref[1])
    sc.close()


def test_tiles_of_a_mixed_batch_and_of_a_reused_frame(ctx, pool):
    """A batch of images and a ray list in one call; then a second frame of a
    static camera with one part moved, its hits reused."""
    import torch

    import paper_1911_06001_gb300 as g

    made = [_scene(ctx, pool, p, 300 + p) for p in (5, 70, 130)]
    sizes = [(200, 163), (257, 140), (0, 0)]
    rays = [_rays("pinhole", w, h, s.meta["box"], 7) if w else _rays("incoherent", 100, 51, s.meta["box"], 8)
            for (_, s), (w, h) in zip(made, sizes)]
    ref = [_trace(sc, r, g.TRACE_DEFAULT) for (sc, _), r in zip(made, rays)]
    dev = [torch.from_numpy(r).cuda() for r in rays]
    hits = [torch.empty((r.shape[0], 2), dtype=torch.int64, device="cuda") for r in dev]
    rfs = [torch.full((r.shape[0],), 77, dtype=torch.int32, device="cuda") for r in dev]
    ctx.trace_batch([(sc, r, h, f, w) for (sc, _), r, h, f, (w, _) in zip(made, dev, hits, rfs, sizes)])
    torch.cuda.synchronize()
    for h, f, want in zip(hits, rfs, ref):
        assert np.array_equal(h.cpu().numpy(), want[0]) and np.array_equal(f.cpu().numpy(), want[1])
    sc, s = made[1]
    w = sizes[1][0]
    flags = g.TRACE_DEFAULT | g.trace_image(w)
    _trace(sc, rays[1], flags, hits[1])
    local = s.local.copy()
    local[3, 3::4] += 0.2
    sc.set_transforms(local)
    sc.refit()
    got = _trace(sc, rays[1], flags | g.TRACE_REUSE, hits[1])
    ref2 = _trace(sc, rays[1], g.TRACE_DEFAULT)
    assert np.array_equal(got[0], ref2[0])
    assert (got[1] == g.RAY_REUSED).sum() > 100
    for sc, _ in made:
        sc.close()
