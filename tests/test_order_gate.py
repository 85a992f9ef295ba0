"""Rays to be ordered by origin around the limits of the shapes such a call
takes -- few and many rays, fewer than 128 parts and more, few, some and all
rays meeting a part: hits and flags equal those of the plain call bit for bit,
call after call on one stream."""

from __future__ import annotations

import numpy as np
import pytest

import synthetic

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("parts", [1, 16, 127, 128])
@pytest.mark.parametrize("n", [(1 << 18) - 1, 1 << 18, 300_001])
def test_shapes(parts, n):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__

    __graft_entry__.build()
    import paper_1911_06001_gb300 as g

    ctx = g.Context(0)
    pool = synthetic.asset_pool(range(4, 6), 2, seed=4)
    s = synthetic.batched_scenes(seed=parts, n_scenes=1, parts=(parts, parts), depths=range(4, 6), side=(8, 9),
                                 per_depth=2, pool=pool).scenes[0]
    sc = ctx.scene([ctx.upload(a.asset.depth, a.asset.leaf_ids, a.asset.rgb) for a in
                    (pool[int(a)] for a in s.part_asset)], s.parent)
    sc.set_transforms(s.local)
    sc.refit()
    rng = np.random.default_rng(n + parts)
    mid = sc.read_poses()["sphere"][:, :3][rng.integers(0, parts, n)].astype(np.float64)
    out = rng.standard_normal((n, 3))
    out *= 3.0 * s.meta["box"] / np.linalg.norm(out, axis=1, keepdims=True)  # outside the scene
    for met in (0.0, 0.375 + parts / 205.0 - 0.05, 0.375 + parts / 205.0 + 0.05, 1.0):
        rays = np.zeros((n, 8), np.float32)
        rays[:, :3] = mid + out
        rays[:, 4:7] = np.where((rng.random(n) < met)[:, None], -out, out)  # towards a part, or away
        rays[:, 7] = np.inf
        r = torch.from_numpy(rays).cuda()
        ref = None
        for flags in (0, g.TRACE_ORDER_ORIGIN, g.TRACE_ORDER_ORIGIN | g.TRACE_DEFER_FIX, g.TRACE_ORDER_ORIGIN):
            rf = torch.full((n,), 77, dtype=torch.int32, device="cuda")
            hits = sc.trace(r, flags=g.TRACE_DEFAULT | flags, ray_flags=rf)
            ctx.fix_pending()
            torch.cuda.synchronize()
            if ref is None:
                ref = hits, rf
            assert torch.equal(hits, ref[0]) and torch.equal(rf, ref[1]), (met, flags)
    ctx.check_device()
    sc.close()
    ctx.close()
