"""A stream's launch counters are ready whether its first call runs eagerly or
is captured: a call that is only recorded leaves nothing undone for an eager
call before the first replay."""

from __future__ import annotations

import numpy as np
import pytest

import synthetic

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("form", ["fix", "image", "wave", "origin", "no_fix", "defer"])
def test_first_call_of_a_stream_captured(form):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__

    __graft_entry__.build()
    import paper_1911_06001_gb300 as g

    ctx = g.Context(0)
    pool = synthetic.asset_pool(range(6, 8), 2, seed=9)
    s = synthetic.batched_scenes(seed=3, n_scenes=1, parts=(40, 40), depths=range(6, 8), side=(64, 65), per_depth=2,
                                 pool=pool).scenes[0]
    sc = ctx.scene([ctx.upload(a.asset.depth, a.asset.leaf_ids, a.asset.rgb) for a in
                    (pool[int(a)] for a in s.part_asset)], s.parent)
    sc.set_transforms(s.local)
    sc.refit()
    w, h = 192, 128
    rays = torch.from_numpy(synthetic.pinhole_rays(np.array([0.2, 0.3, 1.0]) * s.meta["box"], (0, 0, 0), w, h)).cuda()
    flags = {"fix": 0, "image": g.trace_image(w), "wave": g.TRACE_WAVEFRONT, "origin": g.TRACE_ORDER_ORIGIN,
             "no_fix": 0, "defer": g.TRACE_DEFER_FIX}[form] | (g.TRACE_CULL | g.TRACE_SORT if form == "no_fix"
                                                                else g.TRACE_DEFAULT)
    ref = sc.trace(rays, flags=flags & ~(g.TRACE_WAVEFRONT | g.TRACE_ORDER_ORIGIN | g.TRACE_DEFER_FIX))
    # memory that the stream's counters may get holds no zeros
    torch.full((1 << 22,), -1, dtype=torch.int64, device="cuda")
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    stream = torch.cuda.Stream()
    hits = torch.zeros((w * h, 2), dtype=torch.int64, device="cuda")
    graph = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph, stream=stream, capture_error_mode="relaxed"):
        sc.trace(rays, hits, flags=flags)
        ctx.fix_pending()
    for replay in (False, True, False, True):
        hits.fill_(-7)
        with torch.cuda.stream(stream):
            stream.wait_stream(torch.cuda.default_stream())
            if replay:
                graph.replay()
            else:
                sc.trace(rays, hits, flags=flags)
                ctx.fix_pending()
        torch.cuda.synchronize()
        assert torch.equal(hits, ref), (form, replay)
    ctx.check_device()
    del graph
    sc.close()
    ctx.close()
