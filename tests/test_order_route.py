"""Rays to be ordered by origin are traced in the wavefront shape, or by the
single launch where most of them meet a part: for few, about half and all
rays meeting one, hits and flags equal those of the plain call bit for bit,
call after call."""

from __future__ import annotations

import numpy as np
import pytest

import synthetic

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 33, 4096, 70_001])
@pytest.mark.parametrize("met", [0.0, 0.2, 0.49, 0.5, 0.51, 1.0])
def test_order_by_origin(met, n):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__

    __graft_entry__.build()
    import paper_1911_06001_gb300 as g

    ctx = g.Context(0)
    s = synthetic.pr1_scene(depth=5, noise_p=0.0)
    sc = ctx.scene([ctx.upload(a.depth, a.leaf_ids, a.rgb) for a in s.assets], s.parent)
    sc.set_transforms(s.local)
    sc.refit()
    rng = np.random.default_rng(n)
    rays = np.zeros((n, 8), np.float32)
    o = rng.standard_normal((n, 3))
    o *= 6.0 / np.linalg.norm(o, axis=1, keepdims=True)
    rays[:, :3] = o
    aim = rng.uniform(-0.2, 0.2, (n, 3)) - o  # into the root part's sphere
    rays[:, 4:7] = np.where((rng.permutation(n) < round(met * n))[:, None], aim, -aim)  # or away from everything
    rays[:, 7] = np.inf
    r = torch.from_numpy(rays).cuda()
    out = []
    for flags in (0, g.TRACE_ORDER_ORIGIN, g.TRACE_ORDER_ORIGIN, g.TRACE_ORDER_ORIGIN | g.TRACE_DEFER_FIX, 0):
        rf = torch.full((n,), 77, dtype=torch.int32, device="cuda")
        hits = sc.trace(r, flags=g.TRACE_DEFAULT | flags, ray_flags=rf)
        ctx.fix_pending()
        torch.cuda.synchronize()
        out.append((hits.cpu().numpy(), rf.cpu().numpy()))
    for h, f in out[1:]:
        assert np.array_equal(h, out[0][0]) and np.array_equal(f, out[0][1])
    ctx.check_device()
    sc.close()
    ctx.close()
