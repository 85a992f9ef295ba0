"""The descent over the whole range of octree depths: sparse assets whose
leaves sit at the cube's corners, edges and random cells, rays aimed at them
from every octant, against the FP64 oracle element by element."""

from __future__ import annotations

import numpy as np
import pytest

import oracle
import synthetic
from gpu_helpers import GpuScene, compare

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


@pytest.mark.parametrize("depth", [1, 2, 3, 9, 15, 16])
def test_depths(ctx, depth):
    import paper_1911_06001_gb300 as g

    rng = np.random.default_rng(depth)
    n = 1 << depth
    edge = np.array([0, n // 2, n - 1])
    xyz = np.concatenate([np.stack(np.meshgrid(edge, edge, edge), -1).reshape(-1, 3), rng.integers(0, n, (200, 3))])
    asset = synthetic.make_asset(depth, tuple(xyz.T))
    pose = synthetic.affine12(synthetic.euler_xyz(0.3, -0.7, 1.1) * 1.5, (0.2, -0.4, 0.3))
    scene = synthetic.Scene("depths", [asset], np.zeros(2, np.int32), np.array([-1, -1], np.int32),
                            np.stack([pose, synthetic.affine12(np.eye(3), (1.5, 0.0, 0.0))]))
    # to a point of a random leaf of either part, from a point outside
    m = 6000
    part = rng.integers(0, 2, m)
    leaf = np.stack(synthetic.unpack_ids(asset.leaf_ids, depth), 1)[rng.integers(0, asset.n_leaves, m)]
    local = (leaf + rng.random((m, 3))) / n
    w = scene.local.reshape(2, 3, 4)[part]
    target = np.einsum("nij,nj->ni", w[:, :, :3], local) + w[:, :, 3]
    origin = rng.uniform(-4.0, 4.0, (m, 3))
    rays = np.zeros((m, 8), np.float32)
    rays[:, :3], rays[:, 4:7], rays[:, 7] = origin, target - origin, np.inf
    gs = GpuScene(ctx, scene)
    ora = oracle.SceneOracle(scene).trace(rays)
    for flags in (g.TRACE_DEFAULT, g.TRACE_DEFAULT | g.TRACE_WAVEFRONT):
        rep = compare(scene, scene.local, rays, gs.trace(rays, flags), ora)
        assert rep["hits"] > (4000 if depth <= 9 else 1000)
