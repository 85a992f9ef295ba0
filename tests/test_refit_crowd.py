"""Batched refits of many large scenes, whose clusters of blocks shrink with
their number: scene counts on both sides of each limit, alike and mixed with
small scenes, give the bytes of single refits."""

from __future__ import annotations

import numpy as np
import pytest

import synthetic

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sizes", [[600] * 12, [600] * 13, [140] * 32, [140] * 33, [1024] * 13 + [7] * 51,
                                   [1024] * 33 + [300], [70] * 64], ids=lambda s: f"{len(s)}x{max(s)}")
def test_equals_single_refits(sizes):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__

    __graft_entry__.build()
    import paper_1911_06001_gb300 as g

    ctx = g.Context(0)
    pool = synthetic.asset_pool(range(4, 6), 2, seed=5)
    handles = [ctx.upload(p.asset.depth, p.asset.leaf_ids, p.asset.rgb) for p in pool]
    rng = np.random.default_rng(len(sizes))
    batch, local = [], []
    for P in sizes:
        parent = np.array([-1] + [int(rng.integers(max(0, i - 40), i)) if rng.random() < 0.7 else -1
                                  for i in range(1, P)], dtype=np.int32)
        assets = [handles[int(a)] for a in rng.integers(0, len(handles), P)]
        batch.append((ctx.scene(assets, parent), ctx.scene(assets, parent)))
        a = synthetic.euler_xyz(*rng.uniform(-np.pi, np.pi, 3)) @ np.diag(rng.uniform(0.8, 1.2, 3))
        local.append(np.array([synthetic.affine12(a, t) for t in rng.uniform(-3.0, 3.0, (P, 3))]))
    for (one, _), m in zip(batch, local):
        one.set_transforms(m)
        one.refit()
    ctx.refit_batch([b for _, b in batch], [torch.from_numpy(m).cuda() for m in local])
    torch.cuda.synchronize()
    for one, b in batch:
        p, q = ({**sc.read_poses(), **{"c_" + k: v for k, v in sc.read_clusters().items()}} for sc in (one, b))
        for k in p:
            assert np.array_equal(p[k].view(np.uint8), q[k].view(np.uint8)), k
        one.close()
        b.close()
    ctx.check_device()
    ctx.close()
