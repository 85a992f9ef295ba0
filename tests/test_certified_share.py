"""What FP32 alone certifies: on rays that graze leaf faces or frame deep parts
behind transform chains, a trace without the FP64 pass flags no more rays as
uncertain and names no more wrong leaves than it did with corners held in
[0, 1) (its counts on the same rays), and no wrong leaf goes unflagged."""

from __future__ import annotations

import numpy as np
import pytest

import oracle
import synthetic

pytestmark = pytest.mark.gpu

# (seed, depth) -> uncertain rays, wrong leaves, of 60,000
COUNTS = {(50, 13): (27916, 12835), (50, 9): (11164, 5428), (51, 13): (28087, 12919), (51, 9): (11773, 5752),
          (52, 13): (28519, 13273), (52, 9): (11424, 5611)}


@pytest.mark.parametrize("seed,depth", COUNTS)
def test_uncertain_and_wrong(seed, depth):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__

    __graft_entry__.build()
    import paper_1911_06001_gb300 as g

    prec = synthetic.precision_scene(seed=seed, n_visible=4, chain=3, depth=depth,
                                     radius=(20.0, 60.0) if depth == 9 else (100.0, 250.0),
                                     max_shift_leaves=1e3 if depth == 9 else 1e4)
    s = prec.scene
    rays, _ = synthetic.precision_rays(prec, oracle.compose(s.parent, s.local), n_total=60_000, graze_frac=0.5, seed=seed)
    ctx = g.Context(0)
    handles = [ctx.upload(a.depth, a.leaf_ids, a.rgb) for a in s.assets]
    sc = ctx.scene([handles[int(a)] for a in s.part_asset], s.parent)
    sc.set_transforms(s.local)
    sc.refit()
    rf = torch.zeros(len(rays), dtype=torch.int32, device="cuda")
    hits = g.decode_hits(sc.trace(torch.from_numpy(rays).cuda(), flags=g.TRACE_CULL | g.TRACE_SORT, ray_flags=rf))
    uncertain = (rf.cpu().numpy() & g.RAY_UNCERTAIN) != 0
    ref = oracle.SceneOracle(s).trace(rays)
    wrong = (hits["part"] != ref["part"]) | (hits["voxel"] != ref["voxel"])
    assert not (wrong & ~uncertain).any()
    assert uncertain.sum() <= COUNTS[seed, depth][0]
    assert wrong.sum() <= COUNTS[seed, depth][1]
    ctx.check_device()
    sc.close()
    ctx.close()
