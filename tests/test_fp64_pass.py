"""The FP64 pass on short and long lists: rays that graze leaf faces (lists of
contenders of every length, and rays whose list overflowed) and close pinhole
rays (t refinements), alone and over several scenes in one batch, against the
FP64 oracle element by element."""

from __future__ import annotations

import numpy as np
import pytest

import oracle
import synthetic
from gpu_helpers import compare

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


@pytest.mark.parametrize("n", [120, 700, 60_000])
@pytest.mark.parametrize("depth", [9, 13])
def test_flagged_rays(ctx, depth, n):
    import torch

    import paper_1911_06001_gb300 as g

    made, items = [], []
    for k in range(3):
        prec = synthetic.precision_scene(seed=50 + k, n_visible=4, chain=3, depth=depth,
                                         radius=(20.0, 60.0) if depth == 9 else (100.0, 250.0), max_shift_leaves=1e3)
        s = prec.scene
        world = oracle.compose(s.parent, s.local)
        m = max(n // 3, 10)
        rays, _ = synthetic.precision_rays(prec, world, n_total=m, graze_frac=0.8, seed=k)
        handles = [ctx.upload(a.depth, a.leaf_ids, a.rgb) for a in s.assets]
        sc = ctx.scene([handles[int(a)] for a in s.part_asset], s.parent)
        sc.set_transforms(s.local)
        sc.refit()
        made.append((sc, s, rays, oracle.SceneOracle(s).trace(rays)))
        r = torch.from_numpy(rays).cuda()
        items.append((sc, r, torch.empty((len(rays), 2), dtype=torch.int64, device="cuda"),
                      torch.zeros(len(rays), dtype=torch.int32, device="cuda")))

    def check(k, hits, rf):
        sc, s, rays, ora = made[k]
        out = g.decode_hits(hits)
        out["flags"] = rf.cpu().numpy().astype(np.uint32)
        return compare(s, s.local, rays, out, ora)

    fixed = 0
    for k, (sc, r, _, _) in enumerate(items):
        rf = torch.zeros(r.shape[0], dtype=torch.int32, device="cuda")
        hits = sc.trace(r, ray_flags=rf)
        torch.cuda.synchronize()
        fixed += check(k, hits, rf)["fixed"]
    ctx.trace_batch(items)
    torch.cuda.synchronize()
    assert sum(check(k, it[2], it[3])["fixed"] for k, it in enumerate(items)) == fixed
    assert fixed > n // 4
    for sc, *_ in made:
        sc.close()
