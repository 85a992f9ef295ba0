"""One scene traced from several streams at once, each ordered after the refit
that made its grid stale: the call forms that walk the scene grid share its
one copy, and every stream's hits and flags equal those of the plain call."""

from __future__ import annotations

import numpy as np
import pytest

import synthetic

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("parts", [64, 333, 1024])
def test_traces_of_one_scene_on_three_streams(parts):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__

    __graft_entry__.build()
    import paper_1911_06001_gb300 as g

    ctx = g.Context(0)
    pool = synthetic.asset_pool(range(5, 7), 2, seed=4)
    handles = [ctx.upload(a.asset.depth, a.asset.leaf_ids, a.asset.rgb) for a in pool]
    s = synthetic.batched_scenes(seed=parts, n_scenes=1, parts=(parts, parts), depths=range(5, 7), side=(8, 9),
                                 per_depth=2, pool=pool).scenes[0]
    sc = ctx.scene([handles[int(a)] for a in s.part_asset], s.parent)
    box = s.meta["box"]
    n = (1 << 25) // parts + 77  # enough rays for the wavefront shape to use the grid
    rays = torch.from_numpy(synthetic.random_rays(n, np.random.default_rng(parts), (-box / 2,) * 3,
                                                  (box / 2,) * 3)).cuda()
    streams = [torch.cuda.Stream() for _ in range(3)]
    forms = [g.TRACE_WAVEFRONT, g.TRACE_ORDER_ORIGIN, g.TRACE_GRID]
    hits = [torch.empty((n, 2), dtype=torch.int64, device="cuda") for _ in forms]
    rfs = [torch.empty(n, dtype=torch.int32, device="cuda") for _ in forms]
    turn = np.eye(3)
    for k in range(24):
        turn = synthetic.euler_xyz(0.3, 0.5, -0.2) @ turn
        local = s.local.reshape(-1, 3, 4)
        local = np.concatenate([turn @ local[:, :, :3], turn @ local[:, :, 3:]], 2).reshape(-1, 12)
        sc.set_transforms(local)
        sc.refit()
        ref_f = torch.empty(n, dtype=torch.int32, device="cuda")
        ref = sc.trace(rays, flags=g.TRACE_DEFAULT, ray_flags=ref_f)
        for st, form, h, f in zip(streams, forms[k % 3:] + forms[:k % 3], hits, rfs):
            h.fill_(-7)
            st.wait_stream(torch.cuda.current_stream())
            sc.trace(rays, h, flags=g.TRACE_DEFAULT | form, ray_flags=f, stream=st)
        torch.cuda.synchronize()
        for h, f in zip(hits, rfs):
            assert torch.equal(h, ref) and torch.equal(f, ref_f), k
    ctx.check_device()
    sc.close()
    ctx.close()
