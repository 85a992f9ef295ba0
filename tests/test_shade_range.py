"""Shading over the range where its FP32 decisions give way to FP64 ones: deep
leaves, scenes far from the origin, rays that start inside a leaf, graze an
edge or run along an axis, lights from behind -- every pixel the FP64 oracle
calls unambiguous is equal."""

from __future__ import annotations

import numpy as np
import pytest

import oracle
import synthetic
from gpu_helpers import GpuScene
from test_gpu_parity import _shade_case

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


@pytest.mark.parametrize("depth,scale,offset", [(4, 1.0, 0.0), (9, 1.0, 0.0), (9, 50.0, 1e3), (7, 1e-3, 2.0),
                                                (8, 2.0, 3e4), (12, 1.0, 0.0)])
def test_shade(ctx, depth, scale, offset):
    rng = np.random.default_rng(depth)
    n = 1 << depth
    cells = synthetic.ellipsoid_shell(depth, (n / 2,) * 3, np.array([0.3, 0.22, 0.4]) * min(n, 512), 1.0)
    asset = synthetic.make_asset(depth, cells)
    a = synthetic.euler_xyz(0.4, 0.9, -0.3) @ np.diag([1.0, 0.7, 1.3]) * scale
    t = np.array([0.3, -0.2, 0.1]) * scale + offset
    scene = synthetic.Scene("shade", [asset], np.zeros(1, np.int32), np.array([-1], np.int32),
                            synthetic.affine12(a, t)[None])
    mid = a @ np.full(3, 0.5) + t
    size = scale * min(1.0, 512 / n)
    rays = synthetic.pinhole_rays(mid + size * np.array([0.4, 0.9, 1.2]), mid, 160, 120, 50.0)
    m = 3000
    inside = (np.stack(synthetic.unpack_ids(asset.leaf_ids, depth), 1)[rng.integers(0, asset.n_leaves, m)]
              + rng.random((m, 3))) / n
    more = np.zeros((m, 8), np.float32)
    more[:, :3] = inside @ a.T + t
    more[:, 4:7] = rng.standard_normal((m, 3))
    more[:, 7] = np.inf
    more[:500, 4:7] = a.T[rng.integers(0, 3, 500)] * rng.choice([-1.0, 1.0], (500, 1))
    more[:500, :3] -= (more[:500, 4:7] * 0.7).astype(np.float32)
    more[500:1500, :3] -= more[500:1500, 4:7] * np.float32(3 * size)
    rays = np.concatenate([rays, more]).astype(np.float32)
    gs = GpuScene(ctx, scene)
    for light, ambient in (((0.3, 0.8, 0.5), 0.2), ((-1.0, -0.2, 0.1), 0.0), ((0.0, 1.0, 0.0), 1.0)):
        hits, amb = _shade_case(ctx, gs, oracle.SceneOracle(scene), rays, light, ambient, 0x102030)
        assert hits > 1500
