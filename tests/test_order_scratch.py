"""Scratch of rays to be ordered by origin: one call at full size makes room for
every route such a call can take, so that later calls of any form can be
captured; where the wavefront shape's queue has no room the rays are sorted."""

from __future__ import annotations

import numpy as np
import pytest

import synthetic

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__

    __graft_entry__.build()
    import paper_1911_06001_gb300 as g

    ctx = g.Context(0)
    pool = synthetic.asset_pool(range(5, 7), 2, seed=9)
    bat = synthetic.batched_scenes(seed=2, n_scenes=2, parts=(70, 90), depths=range(5, 7), side=(64, 65), per_depth=2,
                                   pool=pool)
    scenes, rays = [], []
    for k, s in enumerate(bat.scenes):
        sc = ctx.scene([ctx.upload(a.asset.depth, a.asset.leaf_ids, a.asset.rgb) for a in
                        (pool[int(a)] for a in s.part_asset)], s.parent)
        sc.set_transforms(s.local)
        sc.refit()
        b = s.meta["box"]
        scenes.append(sc)
        rays.append(torch.from_numpy(synthetic.random_rays(40_000, np.random.default_rng(k), (-b,) * 3, (b,) * 3)).cuda())
    yield g, ctx, scenes, rays
    ctx.check_device()
    for sc in scenes:
        sc.close()
    ctx.close()


def _hits(n):
    import torch

    return torch.zeros((n, 2), dtype=torch.int64, device="cuda")


def test_one_warm_call_covers_every_route(env):
    import torch

    g, ctx, scenes, rays = env
    ref = [sc.trace(r) for sc, r in zip(scenes, rays)]
    torch.cuda.synchronize()
    stream = torch.cuda.Stream()
    warm = torch.cat([rays[0], rays[0], rays[0]])[:100_000].contiguous()
    scenes[0].trace(warm, flags=g.TRACE_DEFAULT | g.TRACE_ORDER_ORIGIN, stream=stream)
    got = [_hits(r.shape[0]) for r in rays]
    one, kept = _hits(rays[0].shape[0]), ref[0].clone()
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    f = g.TRACE_DEFAULT | g.TRACE_ORDER_ORIGIN
    with torch.cuda.graph(graph, stream=stream):
        ctx.trace_batch([(sc, r, h, None) for sc, r, h in zip(scenes, rays, got)], flags=f)
        scenes[0].trace(rays[0], one, flags=f)
        scenes[0].trace(rays[0], kept, flags=f | g.TRACE_REUSE)
    graph.replay()
    torch.cuda.synchronize()
    assert all(torch.equal(a, b) for a, b in zip(got, ref))
    assert torch.equal(one, ref[0]) and torch.equal(kept, ref[0])


def test_sorted_where_the_queue_has_no_room(env):
    import torch

    g, _, scenes, rays = env
    ref = scenes[0].trace(rays[0])
    torch.cuda.synchronize()
    stream = torch.cuda.Stream()
    scenes[0].trace(rays[0], flags=g.TRACE_DEFAULT | g.TRACE_ORDER_DIR, stream=stream)  # no queue on this stream
    hits = _hits(rays[0].shape[0])
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream):
        scenes[0].trace(rays[0], hits, flags=g.TRACE_DEFAULT | g.TRACE_ORDER_ORIGIN)
    for _ in range(2):
        hits.zero_()
        torch.cuda.synchronize()
        graph.replay()
        torch.cuda.synchronize()
        assert torch.equal(hits, ref)


def test_warm_call_of_a_small_scene_serves_a_large_one(env):
    import torch

    g, ctx, scenes, rays = env
    n = rays[0].shape[0]
    big = ctx.scene([1] * 200, np.full(200, -1, np.int32))
    big.set_transforms(np.array([synthetic.affine12(np.eye(3), t) for t in
                                 np.random.default_rng(1).uniform(-9.0, 9.0, (200, 3))]))
    big.refit()
    stream, f = torch.cuda.Stream(), g.TRACE_DEFAULT | g.TRACE_ORDER_ORIGIN
    ref = big.trace(rays[0])
    hits = _hits(n)
    torch.cuda.synchronize()
    scenes[0].trace(rays[0], hits, flags=f, stream=stream)
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    big.trace(rays[0], hits, flags=f, stream=stream)
    torch.cuda.synchronize()
    assert torch.cuda.mem_get_info()[0] == free
    assert torch.equal(hits, ref)
    big.close()
