"""The server's bytes per ray cover what the library allocates: device memory
taken by a stream's first call, for the flags a server may be given."""

from __future__ import annotations

import pytest

import synthetic

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("form", ["default", "wavefront", "origin", "dir"])
def test_scratch_per_ray(form):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__

    __graft_entry__.build()
    import paper_1911_06001_gb300 as g
    from paper_1911_06001_gb300 import serving

    flags = g.TRACE_DEFAULT | {"default": 0, "wavefront": g.TRACE_WAVEFRONT, "origin": g.TRACE_ORDER_ORIGIN,
                               "dir": g.TRACE_ORDER_DIR}[form]
    ctx = g.Context(0)
    s = synthetic.pr1_scene(depth=5, noise_p=0.0)
    sc = ctx.scene([ctx.upload(a.depth, a.leaf_ids, a.rgb) for a in s.assets], s.parent)
    sc.set_transforms(s.local)
    sc.refit()
    n = 1 << 23
    rays = torch.zeros((n, 8), dtype=torch.float32, device="cuda")
    rays[:, 7] = -1.0  # empty segments
    hits = torch.empty((n, 2), dtype=torch.int64, device="cuda")
    sc.trace(rays[:64], hits[:64], flags=flags)  # kernels and the smallest scratch are there
    torch.cuda.synchronize()
    stream = torch.cuda.Stream()
    before = torch.cuda.mem_get_info()[0]
    ctx.trace_batch([(sc, rays, hits, None)], flags=flags, stream=stream)
    torch.cuda.synchronize()
    used = before - torch.cuda.mem_get_info()[0]
    # allocations are rounded to 2 MiB each; at most six of them
    assert used <= n * serving.scratch_bytes_per_ray(flags) + 6 * (2 << 20)
    assert used >= n * (serving.scratch_bytes_per_ray(flags) - 10)
    sc.close()
    ctx.close()
