"""Image traces through the scene grid whose tiles have no part list -- more
parts than a list holds, or rays that no cone bounds -- walk the grid: in scenes
of touching parts, seen whole and from inside, singly and in a batch with a
scene that has no grid, hits and flags equal those of the plain call."""

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
def model(ctx):
    n = 32
    a = synthetic.make_asset(5, synthetic.ellipsoid_shell(5, (n / 2,) * 3, (0.48 * n,) * 3, 1.5))
    return ctx.upload(a.depth, a.leaf_ids, a.rgb)


def _lattice(ctx, model, k):
    local = np.array([synthetic.affine12(synthetic.euler_xyz(0.1 * x, 0.2 * y, 0.3 * z),
                                         np.array([x, y, z]) - k / 2) for x in range(k) for y in range(k)
                      for z in range(k)])
    sc = ctx.scene([model] * k ** 3, np.full(k ** 3, -1, np.int32))
    sc.set_transforms(local)
    sc.refit()
    return sc, local


def _image(k, view, w, h):
    eye = np.array([0.9, 1.1, 1.6]) * k if view == "whole" else np.array([0.13, 0.15, 0.19]) * k
    rays = synthetic.pinhole_rays(eye, (0.0, 0.0, 0.0), w, h, 60.0 if view == "whole" else 100.0)
    if view == "behind":
        rays[::5, 3] = -0.7 * k
    return rays.astype(np.float32)


@pytest.mark.parametrize("view", ["whole", "inside", "behind"])
@pytest.mark.parametrize("k", [3, 4, 5, 10])
def test_touching_parts(ctx, model, k, view):
    import torch

    import paper_1911_06001_gb300 as g

    sc, local = _lattice(ctx, model, k)
    w, h = 331, 173
    r = torch.from_numpy(_image(k, view, w, h)).cuda()
    for turn in range(3):  # the grid stale, built, and stale again
        if turn == 2:
            sc.set_transforms(local)
            sc.refit()
        out = []
        for flags in (0, g.trace_image(w) | g.TRACE_GRID):
            rf = torch.full((w * h,), 77, dtype=torch.int32, device="cuda")
            out.append((sc.trace(r, flags=g.TRACE_DEFAULT | flags, ray_flags=rf), rf))
        torch.cuda.synchronize()
        assert torch.equal(out[0][0], out[1][0]) and torch.equal(out[0][1], out[1][1]), turn
    sc.close()


def test_batch_of_images(ctx, model):
    import torch

    import paper_1911_06001_gb300 as g

    made = [(_lattice(ctx, model, k)[0], _image(k, v, 200, 120)) for k, v in ((3, "whole"), (10, "whole"), (6, "inside"),
                                                                              (2, "whole"))]
    out = []
    for flags, width in ((0, 0), (g.TRACE_GRID, 200)):
        items = [(sc, torch.from_numpy(r).cuda(), torch.empty((len(r), 2), dtype=torch.int64, device="cuda"),
                  torch.full((len(r),), 77, dtype=torch.int32, device="cuda"), width) for sc, r in made]
        ctx.trace_batch(items, flags=g.TRACE_DEFAULT | flags)
        torch.cuda.synchronize()
        out.append(items)
    for a, b in zip(*out):
        assert torch.equal(a[2], b[2]) and torch.equal(a[3], b[3])
    for sc, _ in made:
        sc.close()
