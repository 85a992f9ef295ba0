"""Shading of parts whose transforms cancel: rays aimed at leaf edges of deep
parts far from the world's origin (and of small and near ones).  A pixel the FP32
decisions settle gets the bytes of the FP64 way, which the same rays take with
tmin = -inf: no start inside the leaf can then be told apart from FP32, and the
FP64 rule itself does not depend on it for rays entered from outside."""

from __future__ import annotations

import numpy as np
import pytest

import synthetic

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("depth,scale,offset", [(6, 1.0, 0.0), (13, 1.0, 0.0), (13, 1.0, 2.0 ** 17), (13, 1.0, 2.0 ** 27),
                                                (16, 1.0, 2.0 ** 22), (9, 2.0 ** -10, 2.0 ** 12),
                                                (11, 2.0 ** 10, 2.0 ** 27)])
def test_far_parts(depth, scale, offset):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__

    __graft_entry__.build()
    import paper_1911_06001_gb300 as g

    rng = np.random.default_rng(depth)
    n = 1 << depth
    cells = np.unique(rng.integers(0, n, (4000, 3)), axis=0)
    asset = synthetic.make_asset(depth, tuple(cells.T))
    a = synthetic.euler_xyz(0.4, 0.9, -0.3) * scale
    t = np.array([1.0, -0.5, 0.25]) * offset
    ctx = g.Context(0)
    sc = ctx.scene([ctx.upload(asset.depth, asset.leaf_ids, asset.rgb)], [-1])
    sc.set_transforms(synthetic.affine12(a, t)[None])
    sc.refit()

    m = 200_000
    cell = cells[rng.integers(0, len(cells), m)]
    # a point on an edge of the leaf: two coordinates on its faces, the third inside
    on = rng.integers(0, 2, (m, 3)).astype(np.float64)
    free = rng.integers(0, 3, m)
    on[np.arange(m), free] = rng.uniform(0.1, 0.9, m)
    p = ((cell + on) / n) @ a.T + t
    # looking at that edge from outside the leaf, both of its faces turned to the viewer
    away = np.where(on > 0.5, 1.0, -1.0) * rng.uniform(0.3, 1.0, (m, 3))
    away[np.arange(m), free] = rng.uniform(-0.5, 0.5, m)
    away = away @ a.T
    o = (p + away / np.linalg.norm(away, axis=1, keepdims=True) * 16.0 * max(scale, 2.0 ** -23 * offset)).astype(np.float32)
    d = p - o.astype(np.float64)
    rays = np.zeros((m, 8), np.float32)
    rays[:, :3] = o
    rays[:, 4:7] = d / np.linalg.norm(d, axis=1, keepdims=True)
    rays[:, 7] = np.inf
    hits = np.zeros((m, 4), np.uint32)
    hits[:, 0] = np.linalg.norm(d, axis=1).astype(np.float32).view(np.uint32)
    vox = cell[:, 0].astype(np.uint64) | (cell[:, 1].astype(np.uint64) << np.uint64(depth)) | \
        (cell[:, 2].astype(np.uint64) << np.uint64(2 * depth))
    hits[:, 2], hits[:, 3] = (vox & np.uint64(0xFFFFFFFF)).astype(np.uint32), (vox >> np.uint64(32)).astype(np.uint32)
    h = torch.from_numpy(hits.view(np.int64)).cuda()
    exact = rays.copy()
    exact[:, 3] = -np.inf
    for light in ((0.3, 0.8, 0.5), (-0.6, -0.2, 0.7)):
        got, want = (sc.shade(torch.from_numpy(r).cuda(), h, light, 0.2) for r in (rays, exact))
        assert not (want == -1).any()
        assert torch.equal(got, want), int((got != want).sum())
    ctx.check_device()
    sc.close()
    ctx.close()
