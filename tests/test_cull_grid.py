"""The wavefront shape's culling launch walks the scene grid where a scene has
a sparse one: for part counts around the grid's limits, scenes whose grid is
declined (crowded cells, far from the origin), one scene and batches, and rays
of every kind the walk accepts or steps aside for, hits and flags equal those
of the single launch bit for bit."""

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
    p = synthetic.asset_pool(range(5, 7), 2, seed=4)
    return p, [ctx.upload(a.asset.depth, a.asset.leaf_ids, a.asset.rgb) for a in p]


def _scene(ctx, pool, parts, layout):
    s = synthetic.batched_scenes(seed=parts, n_scenes=1, parts=(parts, parts), depths=range(5, 7), side=(8, 9),
                                 per_depth=2, pool=pool[0]).scenes[0]
    local = s.local.reshape(-1, 3, 4).copy()
    if layout == "crowded":
        local[:, :, 3] *= 0.15
    if layout == "far":
        local[:, :, 3] += np.array([3e5, -2e5, 1e5])
    if layout == "flat":
        local[:, 1, 3] = 0.0
    sc = ctx.scene([pool[1][int(a)] for a in s.part_asset], s.parent)
    sc.set_transforms(local.reshape(-1, 12))
    sc.refit()
    mid = local[:, :, 3].mean(0)
    return sc, mid, s.meta["box"]


def _rays(n, mid, box, seed):
    rng = np.random.default_rng(seed)
    r = synthetic.random_rays(n, rng, (-0.6 * box,) * 3, (0.6 * box,) * 3)
    r[:, :3] += mid.astype(np.float32)
    k = n // 8
    r[:k, 4 + rng.integers(0, 3)] = 0.0                     # axis-parallel planes
    r[k:2 * k, 4:7] = np.eye(3, dtype=np.float32)[rng.integers(0, 3, k)] * rng.choice([-2.0, 0.5], (k, 1))
    r[2 * k:3 * k, :3] = (mid + (r[2 * k:3 * k, :3] - mid) * 40.0).astype(np.float32)  # from far away, towards it
    r[2 * k:3 * k, 4:7] = mid - r[2 * k:3 * k, :3] + rng.uniform(-box, box, (k, 3)) / 2
    r[3 * k:4 * k, 7] = rng.uniform(0.0, box, k)            # bounded segments
    r[4 * k:4 * k + 500, 3] = -box                          # reaching behind the origin
    r[4 * k + 500:4 * k + 600, 4:7] = 1e-25                 # not rays
    r[4 * k + 600:4 * k + 700, 0] = np.nan
    r[4 * k + 700:5 * k, 4] *= 1e-30                        # a component the walk's arithmetic cannot take
    return r.astype(np.float32)


def _trace(run, n):
    import torch

    hits = [torch.empty((k, 2), dtype=torch.int64, device="cuda") for k in n]
    rfs = [torch.full((k,), 77, dtype=torch.int32, device="cuda") for k in n]
    run(hits, rfs)
    torch.cuda.synchronize()
    return [(h.cpu().numpy(), f.cpu().numpy()) for h, f in zip(hits, rfs)]


@pytest.mark.parametrize("layout", ["sparse", "crowded", "far", "flat"])
@pytest.mark.parametrize("parts", [15, 16, 17, 64, 100, 333, 1024])
def test_one_scene(ctx, pool, parts, layout):
    import torch

    import paper_1911_06001_gb300 as g

    sc, mid, box = _scene(ctx, pool, parts, layout)
    n = max((1 << 25) // parts, 32 * parts) + 77  # just enough rays for the grid, a ragged last tile
    r = torch.from_numpy(_rays(n, mid, box, parts)).cuda()
    ref, got = (_trace(lambda h, f: sc.trace(r, h[0], flags=g.TRACE_DEFAULT | x, ray_flags=f[0]), [n])[0]
                for x in (0, g.TRACE_WAVEFRONT))
    assert np.array_equal(ref[0], got[0]) and np.array_equal(ref[1], got[1])
    sc.close()


def test_batch_of_scenes_with_and_without_grids(ctx, pool):
    import torch

    import paper_1911_06001_gb300 as g

    made = [_scene(ctx, pool, p, lay) for p, lay in ((5, "sparse"), (200, "sparse"), (64, "crowded"), (300, "flat"),
                                                     (1024, "sparse"), (40, "far"))]
    n = [3001, 90_007, 40_000, 9600, 100, 33_333]  # 100 rays against 1024 parts: not worth its grid
    rays = [torch.from_numpy(_rays(max(k, 8000), mid, box, k)[:k]).cuda() for k, (_, mid, box) in zip(n, made)]

    def batch(flags):
        return lambda hits, rfs: ctx.trace_batch([(sc, r, h, f) for (sc, _, _), r, h, f in
                                                  zip(made, rays, hits, rfs)] * 1, flags=flags)

    for extra in (0, g.TRACE_ORDER_ORIGIN):
        ref, got = (_trace(batch(g.TRACE_DEFAULT | x), n) for x in (0, g.TRACE_WAVEFRONT | extra))
        for a, b in zip(ref, got):
            assert np.array_equal(a[0], b[0]) and np.array_equal(a[1], b[1])
    for sc, _, _ in made:
        sc.close()
