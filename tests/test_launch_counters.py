"""Launch counters and pose-change flags are left clean by the FP64 pass and
cleared by the calls that run none: any sequence of call forms on one stream
-- with, without and with a deferred FP64 pass, every launch shape, graph
replays in between -- gives the results each call gives by itself."""

from __future__ import annotations

import numpy as np
import pytest

import synthetic

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("seed", [1, 2, 3])
def test_sequences_of_calls(seed):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__

    __graft_entry__.build()
    import paper_1911_06001_gb300 as g
    from paper_1911_06001_gb300.graphs import BatchGraph

    ctx = g.Context(0)
    pool = synthetic.asset_pool(range(6, 8), 2, seed=9)
    handles = [ctx.upload(a.asset.depth, a.asset.leaf_ids, a.asset.rgb) for a in pool]
    bat = synthetic.batched_scenes(seed=seed, n_scenes=3, parts=(20, 70), depths=range(6, 8), side=(64, 128),
                                   per_depth=2, pool=pool)
    scenes, rays, w = [], [], 128
    for s in bat.scenes:
        sc = ctx.scene([handles[int(a)] for a in s.part_asset], s.parent)
        sc.set_transforms(s.local)
        sc.refit()
        scenes.append(sc)
        eye = np.array([0.2, 0.3, 1.0]) * s.meta["box"]
        rays.append(torch.from_numpy(synthetic.pinhole_rays(eye, (0, 0, 0), w, 96)).cuda())
    image = g.trace_image(w)
    forms = {"fix": 0, "image": image, "wave": g.TRACE_WAVEFRONT, "grid": g.TRACE_GRID, "origin": g.TRACE_ORDER_ORIGIN,
             "defer": g.TRACE_DEFER_FIX, "defer_image": g.TRACE_DEFER_FIX | image}
    n = [r.shape[0] for r in rays]

    def fresh():
        return ([torch.zeros((k, 2), dtype=torch.int64, device="cuda") for k in n],
                [torch.zeros(k, dtype=torch.int32, device="cuda") for k in n])

    def call(form, fix, k, hits, rfs):
        flags = (g.TRACE_DEFAULT if fix else g.TRACE_CULL | g.TRACE_SORT) | forms[form]
        if k == 3:
            width = w if form.endswith("image") else 0
            ctx.trace_batch([(s, r, h, f, width) for s, r, h, f in zip(scenes, rays, hits, rfs)],
                            flags=flags & 0xFFFF & ~g.TRACE_IMAGE_TILES)
        else:
            scenes[k].trace(rays[k], hits[k], flags=flags, ray_flags=rfs[k])

    ref = {}
    for fix in (True, False):  # each call by itself, from zeroed counters of a new stream
        hits, rfs = fresh()
        st = torch.cuda.Stream()
        with torch.cuda.stream(st):
            st.wait_stream(torch.cuda.default_stream())
            for k in range(3):
                call("fix", fix, k, hits, rfs)
        st.synchronize()
        ref[fix] = [(h.cpu().numpy(), f.cpu().numpy()) for h, f in zip(hits, rfs)]

    graph_hits, graph_rfs = fresh()
    graph = BatchGraph(ctx, [(s, r, h, f, w) for s, r, h, f in zip(scenes, rays, graph_hits, graph_rfs)],
                       [s.local for s in bat.scenes])
    rng = np.random.default_rng(seed)
    for _ in range(40):
        form, fix, k = str(rng.choice(list(forms))), bool(rng.random() < 0.7), int(rng.integers(4))
        hits, rfs = fresh()
        call(form, fix, k, hits, rfs)
        done = fix
        if fix and form.startswith("defer"):
            done = bool(rng.random() < 0.5)  # else the pass is dropped by the next call
            if done:
                ctx.fix_pending()
        if rng.random() < 0.2:
            graph.replay()
            torch.cuda.current_stream().wait_stream(graph.stream)
        torch.cuda.synchronize()
        for q in range(3) if k == 3 else (k,):
            h, f = hits[q].cpu().numpy(), rfs[q].cpu().numpy()
            assert np.array_equal(h, ref[done][q][0]), (form, fix, k, done)
            assert np.array_equal(f, ref[done][q][1]), (form, fix, k, done)
    torch.cuda.synchronize()
    for h, f, want in zip(graph_hits, graph_rfs, ref[True]):
        if h.any():
            assert np.array_equal(h.cpu().numpy(), want[0]) and np.array_equal(f.cpu().numpy(), want[1])
    ctx.check_device()
    for sc in scenes:
        sc.close()
    ctx.close()
