"""Refits by a cluster of blocks (scenes of more than 64 parts): poses, spheres
and the sphere hierarchy at part counts around the clusters' sizes, alone and
in a batch, against the FP64 oracle and against the same parts composed as
separate small scenes."""

from __future__ import annotations

import numpy as np
import pytest

import oracle
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


def _poses(P, seed):
    rng = np.random.default_rng(seed)
    local = np.zeros((P, 12))
    for i in range(P):
        a = synthetic.axis_angle(rng.standard_normal(3), rng.uniform(0, 3)) @ np.diag(rng.uniform(0.8, 1.2, 3))
        local[i] = synthetic.affine12(a, rng.uniform(-1, 1, 3))
    return local


@pytest.mark.parametrize("tree", ["flat", "chains", "random"])
@pytest.mark.parametrize("P", [1, 63, 64, 65, 128, 129, 255, 257, 513, 1000, 1024])
def test_refit(ctx, P, tree):
    rng = np.random.default_rng(P)
    h = ctx.upload(3, synthetic.pack_ids([1, 6], [2, 5], [3, 3], 3))
    parent = np.full(P, -1, np.int32)
    if tree != "flat":
        for i in range(1, P):
            parent[i] = (-1 if i % 12 == 0 else i - 1) if tree == "chains" else int(rng.integers(-1, min(i, 40)))
    local = _poses(P, P)
    world = oracle.compose(parent, local)
    inv = oracle.invert(world)
    sc, other = ctx.scene([h] * P, parent), ctx.scene([h] * P, parent)
    sc.set_transforms(local)
    sc.refit()
    other.set_transforms(local)
    small = ctx.scene([h], [-1])
    ctx.refit_batch([small, other])
    got = sc.read_poses()
    # FP64 rounding of up to 12 composed poses, and of the inverse of a well-conditioned one
    scale = np.abs(world).max(axis=1, keepdims=True) + 1.0
    assert np.all(np.abs(got["world"] - world) <= 1e-13 * scale)
    assert np.all(np.abs(got["inv"] - inv) <= 1e-11 * (np.abs(inv).max(axis=1, keepdims=True) * scale + 1.0))
    # every leaf corner lies in its part's sphere, every part's sphere in its cluster's
    corner = np.array([[x, y, z] for x in (1 / 8, 7 / 8) for y in (2 / 8, 6 / 8) for z in (3 / 8, 4 / 8)])
    w = world.reshape(P, 3, 4)
    pts = np.einsum("pij,kj->pki", w[:, :, :3], corner) + w[:, None, :, 3]
    s = got["sphere"].astype(np.float64)
    assert np.all(np.linalg.norm(pts - s[:, None, :3], axis=2) <= s[:, None, 3])
    cl = sc.read_clusters()
    assert sorted(cl["order"]) == list(range(P))
    for c, o in enumerate(np.array_split(cl["order"], range(8, P, 8))):
        d = np.linalg.norm(s[o, :3] - cl["sphere"][c, :3].astype(np.float64), axis=1) + s[o, 3]
        assert np.all(d <= cl["sphere"][c, 3] * (1 + 1e-12))
    # one launch for many scenes gives the same bits
    got2, cl2 = other.read_poses(), other.read_clusters()
    for k in got:
        assert np.array_equal(got[k], got2[k])
    assert np.array_equal(cl["order"], cl2["order"]) and np.array_equal(cl["sphere"], cl2["sphere"])
    for x in (sc, other, small):
        x.close()
