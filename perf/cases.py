"""Workloads of the ray caster as its users run them, for timing and comparing.

Every case is one call (or one frame's calls) of the public Python layer on
seeded synthetic scenes: poses are set, the scenes refitted, rays traced.  The
shapes are those of the repository's own configurations (small rigid scene,
16-part articulated figure, 64 uneven batched scenes, served requests,
1024-part scenes, deep transform chains) and sizes around them.

Assets are seeded ellipsoid and capsule shells that one context keeps uploaded,
as a program with a model library does; poses, cameras and rays come from the
seed of the state.
"""

from __future__ import annotations

import math

import numpy as np
import torch

import paper_1911_06001_gb300 as svo
from paper_1911_06001_gb300.graphs import BatchGraph

REQUEST_SIZES = ((256, 256), (512, 512), (1280, 720), (1920, 1080), (333, 217))


def listed() -> list:
    return [
        # The smallest call: one frame of a 4-part rigid scene at 128x128 (preview, thumbnail); launches count.
        {"name": "frame_small", "kind": "frame", "parts": 4, "depth": 6, "width": 128, "height": 128, "plain": False},
        # The ordinary frame: a 16-part animated figure of depth-9 models in full HD (the benchmark's frame).
        {"name": "frame_figure_1080p", "kind": "frame", "parts": 16, "depth": 9, "width": 1920, "height": 1080,
         "plain": False},
        # Static camera with a few parts moving: the hit buffer of the previous frame is reused.
        {"name": "static_camera", "kind": "static_camera", "parts": 16, "depth": 9, "width": 1280, "height": 768,
         "moving": 3},
        # One deep model that fills the picture: trace, leaf colours and the shaded image.
        {"name": "model_shaded", "kind": "shaded", "parts": 1, "depth": 11, "width": 1280, "height": 768},
        # A frame of several small scenes replayed as one CUDA graph (an interactive application with many views).
        {"name": "graph_views", "kind": "graph", "scenes": 8, "parts": 24, "width": 301, "height": 199},
        # The largest batch: 64 uneven scenes, incoherent rays (light or sensor simulation).
        {"name": "batch_incoherent", "kind": "batch", "scenes": 64, "parts": 256, "rays": 10_900_003},
        # A server's batch: nine render requests of mixed sizes, rays generated on the device.
        {"name": "served_batch", "kind": "served", "requests": 9, "parts": 128},
        # A crowd: 1024 parts in full HD through the scene grid.
        {"name": "crowd_camera", "kind": "crowd_camera", "parts": 1024, "width": 1920, "height": 1080},
        # Incoherent rays that start inside the crowd, culled in a launch of their own.
        {"name": "crowd_inside", "kind": "crowd_inside", "parts": 1024, "rays": 1_000_003},
        # Incoherent rays against a middle-sized scene, sorted by origin first.
        {"name": "ordered_incoherent", "kind": "ordered", "parts": 128, "rays": 2_097_152},
        # Depth-13 models at the ends of long transform chains, a third of the rays grazing leaf faces.
        {"name": "precision", "kind": "precision", "chains": 8, "rays": 1_048_576},
        # Rays and hits in pinned host memory, through the whole host call.
        {"name": "host_rays", "kind": "host", "parts": 16, "depth": 9, "width": 1280, "height": 720},
    ]


def draw(rng) -> dict:
    def log(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    def image(most):
        w = log(97, 1920)
        return {"width": w, "height": max(61, min(1080, int(w * rng.uniform(0.4, 1.0)), most // w))}

    kind = rng.choice(("frame", "static_camera", "shaded", "graph", "batch", "served", "crowd_camera",
                       "crowd_inside", "ordered", "precision", "host"))
    if kind == "frame":
        return {"kind": kind, "parts": log(2, 63), "depth": rng.randint(6, 10), **image(2_073_600),
                "plain": rng.random() < 0.25}
    if kind == "static_camera":
        parts = log(4, 32)
        return {"kind": kind, "parts": parts, "depth": rng.randint(6, 10), **image(2_073_600),
                "moving": rng.randint(1, max(1, parts // 3))}
    if kind == "shaded":
        return {"kind": kind, "parts": rng.choice((1, 1, log(2, 24))), "depth": rng.randint(7, 11),
                **image(2_073_600)}
    if kind == "graph":
        return {"kind": kind, "scenes": rng.randint(1, 12), "parts": log(4, 64), **image(200_000)}
    if kind == "batch":
        return {"kind": kind, "scenes": rng.randint(2, 64), "parts": log(8, 256), "rays": log(100_000, 10_900_000)}
    if kind == "served":
        return {"kind": kind, "requests": rng.randint(1, 9), "parts": log(16, 128)}
    if kind == "crowd_camera":
        return {"kind": kind, "parts": log(64, 1024), **image(2_073_600)}
    if kind == "crowd_inside":
        return {"kind": kind, "parts": log(64, 1024), "rays": log(50_000, 1_000_000)}
    if kind == "ordered":
        return {"kind": kind, "parts": log(8, 200), "rays": log(100_000, 2_097_152)}
    if kind == "precision":
        return {"kind": kind, "chains": rng.randint(2, 8), "rays": log(50_000, 1_048_576)}
    return {"kind": "host", "parts": log(4, 32), "depth": rng.randint(6, 10), **image(2_073_600)}


def _ray_count(case) -> int:
    if case["kind"] == "served":
        return sum(w * h for w, h in _request_sizes(case))
    if case["kind"] == "graph":
        return case["scenes"] * case["width"] * case["height"]
    return case["rays"] if "rays" in case else case["width"] * case["height"]


def work(case) -> dict:
    """Each ray read (32 B) and each hit written (16 B) once; per ray about a sphere test and a transform."""
    n = _ray_count(case)
    per_ray = {"shaded": 56}.get(case["kind"], 48)  # the shaded image and the colours: 4 B each
    return {"bytes": n * per_ray, "flops": n * 60}


# ------------------------------------------------------------------ assets


def _axes(depth: int, index: int):
    """(semi-axes in cells, whether a capsule, shell thickness) of one model of the library."""
    rng = np.random.default_rng(1000 * depth + index)
    n = 1 << depth
    if depth >= 13:
        return np.full(3, rng.uniform(150.0, 400.0)), False, 1.0
    ax = rng.uniform(0.15, 0.30 if depth >= 11 else 0.45, 3) * n
    return ax, index % 2 == 1, 1.0 if depth >= 11 else 2.0


def _semi(depth: int, index: int) -> np.ndarray:
    ax, capsule, _ = _axes(depth, index)
    if capsule:
        r = min(ax[0], ax[1])
        ax = np.array([r, r, max(ax[2], r)])
    return ax / (1 << depth)


def _leaf_ids(depth: int, index: int) -> torch.Tensor:
    """Voxel ids x | y << D | z << 2D of a centred shell: cells inside the outer body and not inside the inner."""
    ax, capsule, thick = _axes(depth, index)
    n = 1 << depth
    c = n / 2.0

    def half(px, py, a):  # half height of the body over a column (NaN outside)
        if capsule:
            r = min(ax[0], ax[1]) - (ax[0] - a[0])
            rho = r * r - (px - c) ** 2 - (py - c) ** 2
            return torch.where(rho >= 0, max(ax[2] - min(ax[0], ax[1]), 0.0) + rho.clamp_min(0).sqrt(), math.nan)
        q = 1.0 - ((px - c) / a[0]) ** 2 - ((py - c) / a[1]) ** 2
        return torch.where(q >= 0, a[2] * q.clamp_min(0).sqrt(), math.nan)

    g = torch.arange(n, device="cuda", dtype=torch.float64) + 0.5
    lo, hi = max(int(c - ax[:2].max()) - 2, 0), min(int(c + ax[:2].max()) + 2, n)
    x, y = torch.meshgrid(torch.arange(lo, hi, device="cuda"), torch.arange(lo, hi, device="cuda"), indexing="ij")
    x, y = x.reshape(-1), y.reshape(-1)
    ho, hi_ = half(g[x], g[y], ax), half(g[x], g[y], ax - thick)
    out = []
    zo = (torch.ceil(c - ho - 0.5).nan_to_num(1).long(), torch.floor(c + ho - 0.5).nan_to_num(0).long())
    zi = (torch.ceil(c - hi_ - 0.5).nan_to_num(1).long(), torch.floor(c + hi_ - 0.5).nan_to_num(0).long())
    hollow = ~torch.isnan(hi_) & (zi[0] <= zi[1])
    runs = ((zo[0], torch.where(hollow, zi[0] - 1, zo[1])), (torch.where(hollow, zi[1] + 1, zo[1] + 1), zo[1]))
    for z0, z1 in runs:
        cnt = torch.where(torch.isnan(ho), 0, (z1 - z0 + 1).clamp_min(0))
        first = torch.repeat_interleave(z0 - (torch.cumsum(cnt, 0) - cnt), cnt)
        z = first + torch.arange(first.numel(), device="cuda")
        out.append(torch.repeat_interleave(x | (y << depth), cnt) | (z << (2 * depth)))
    return torch.cat(out).unique()


_library: dict = {}


def _context():
    if "ctx" not in _library:
        _library["ctx"] = svo.Context(torch.cuda.current_device())
    return _library["ctx"]


def _handle(asset) -> int:
    """Handle of the model (depth, index), uploaded on first use; None is a link without voxels."""
    if asset not in _library:
        if asset is None:
            depth, ids = 1, np.zeros(0, np.uint64)
        else:
            depth, ids = asset[0], _leaf_ids(*asset).cpu().numpy().astype(np.uint64)
        rgb = ((ids * np.uint64(2654435761)) >> np.uint64(16) & np.uint64(0xFFFFFF)).astype(np.uint32)
        _library[asset] = _context().upload(depth, ids, rgb)
    return _library[asset]


# ------------------------------------------------------------ poses and rays


def _rotation(rng) -> np.ndarray:
    q, r = np.linalg.qr(rng.standard_normal((3, 3)))
    q = q * np.sign(np.diag(r))
    return q if np.linalg.det(q) > 0 else -q


def _swing(axis, angle: float) -> np.ndarray:
    k = np.cross(np.eye(3), axis / np.linalg.norm(axis))
    return np.eye(3) + math.sin(angle) * k + (1.0 - math.cos(angle)) * (k @ k)


def _z_to(v) -> np.ndarray:
    x = np.cross(v, [0.0, 1.0, 0.0] if abs(v[1]) < 0.9 else [1.0, 0.0, 0.0])
    x /= np.linalg.norm(x)
    return np.stack([x, np.cross(v, x), v], 1)


def _row(a, b) -> np.ndarray:
    return np.concatenate([a, np.asarray(b)[:, None]], 1).reshape(12)


def _compose(local, parent) -> np.ndarray:
    world = np.zeros((len(parent), 4, 4))
    for i, p in enumerate(parent):
        m = np.vstack([local[i].reshape(3, 4), [0, 0, 0, 1]])
        world[i] = m if p < 0 else world[p] @ m
    return world


def _figure(rng, assets, branch: int = 6) -> dict:
    """A tree of parts: each hangs from a point on an earlier part's surface and swings about a joint."""
    P = len(assets)
    parent = np.array([-1] + [int(rng.integers(max(0, i - branch), i)) for i in range(1, P)], dtype=np.int32)
    local = np.zeros((P, 12))
    for i in range(P):
        if parent[i] < 0:
            local[i] = _row(np.eye(3), [-0.5] * 3)
            continue
        u = rng.standard_normal(3)
        u /= np.linalg.norm(u)
        a = _z_to(u) @ _swing(rng.standard_normal(3), rng.uniform(-0.5, 0.5))
        joint = np.array([0.5, 0.5, 0.5 - _semi(*assets[i])[2]])
        local[i] = _row(a, 0.5 + u * _semi(*assets[parent[i]]) - a @ joint)
    return {"assets": assets, "parent": parent, "local": local}


def _cloud(rng, parts: int) -> dict:
    """Models of every depth with rotation, scale and shear, spread over a box of side 4 P^(1/3)."""
    box = 4.0 * parts ** (1.0 / 3.0)
    assets, local = [], np.zeros((parts, 12))
    for i in range(parts):
        depth = int(rng.integers(6, 12))
        assets.append((depth, int(rng.integers(2 if depth == 11 else 4))))
        h = np.eye(3)
        h[0, 1], h[0, 2], h[1, 2] = rng.uniform(-0.1, 0.1, 3)
        a = _rotation(rng) @ np.diag(rng.uniform(0.5, 2.0, 3)) @ h
        local[i] = _row(a, rng.uniform(-box / 2, box / 2, 3) - a @ np.full(3, 0.5))
    return {"assets": assets, "parent": np.full(parts, -1, np.int32), "local": local, "box": box}


def _chains(rng, chains: int, length: int = 5) -> dict:
    """Depth-13 models at the ends of rigid chains whose links move by up to 1e4 leaf sizes."""
    assets, parent, local = [], [], []
    for v in range(chains):
        for k in range(length):
            shift = rng.uniform(-1e4, 1e4, 3) / 8192 + (rng.uniform(-3.0, 3.0, 3) if k == 0 else 0.0)
            parent.append(len(parent) - 1 if k else -1)
            local.append(_row(_rotation(rng), shift))
            assets.append((13, v % 2) if k == length - 1 else None)
    return {"assets": assets, "parent": np.array(parent, np.int32), "local": np.array(local)}


def _camera(rng, scene, spread: float = 1.7):
    """(eye, target) seeing the whole scene in a 60 degree field of view from a random side."""
    w = _compose(scene["local"], scene["parent"])
    mid = w[:, :3, :3] @ np.full(3, 0.5) + w[:, :3, 3]
    size = max(np.abs(m[:3, :3]).sum(1).max() for m in w) * 0.4
    target = 0.5 * (mid.min(0) + mid.max(0))
    view = rng.standard_normal(3)
    view /= np.linalg.norm(view)
    return target + view * spread * (np.linalg.norm(mid - target, axis=1).max() + size), target


def _pinhole(eye, target, width: int, height: int, fov: float = 60.0) -> torch.Tensor:
    """Primary rays in 64 bits, row by row."""
    f = np.asarray(target, float) - eye
    f /= np.linalg.norm(f)
    up = np.array([0.0, 1.0, 0.0])
    if abs(up @ f) > 0.999:
        up = np.array([1.0, 0.0, 0.0]) if abs(f[0]) < 0.9 else np.array([0.0, 0.0, 1.0])
    r = np.cross(f, up)
    r /= np.linalg.norm(r)
    f, r, u = (torch.tensor(v, device="cuda", dtype=torch.float64) for v in (f, r, np.cross(r, f)))
    th = math.tan(math.radians(fov) / 2)
    x = (2 * (torch.arange(width, device="cuda", dtype=torch.float64) + 0.5) / width - 1) * th * width / height
    y = (1 - 2 * (torch.arange(height, device="cuda", dtype=torch.float64) + 0.5) / height) * th
    d = f + x[None, :, None] * r + y[:, None, None] * u
    d = (d / d.norm(dim=2, keepdim=True)).reshape(-1, 3)
    rays = torch.zeros((d.shape[0], 8), device="cuda", dtype=torch.float64)
    rays[:, :3] = torch.tensor(np.asarray(eye, float), device="cuda")
    rays[:, 4:7] = d
    rays[:, 7] = math.inf
    return rays


def _incoherent(n: int, box: float, gen) -> torch.Tensor:
    """Origins uniform in the box, directions uniform on the sphere."""
    rays = torch.zeros((n, 8), device="cuda")
    rays[:, :3] = (torch.rand((n, 3), device="cuda", generator=gen) - 0.5) * box
    d = torch.randn((n, 3), device="cuda", generator=gen, dtype=torch.float64)
    rays[:, 4:7] = d / d.norm(dim=1, keepdim=True)
    rays[:, 7] = math.inf
    return rays


def _close_up(rng, gen, scene, n: int) -> torch.Tensor:
    """70% pinhole rays framing each deep model, 30% rays grazing a face of one of its leaves."""
    world = _compose(scene["local"], scene["parent"])
    ends = [i for i, a in enumerate(scene["assets"]) if a is not None]
    side = int(math.sqrt(0.7 * n / len(ends)))
    out, left = [], n - side * side * len(ends)
    for k, i in enumerate(ends):
        w, (depth, _) = world[i], scene["assets"][i]
        c, r = w[:3, :3] @ np.full(3, 0.5) + w[:3, 3], _semi(*scene["assets"][i])[0]
        view = rng.standard_normal(3)
        out.append(_pinhole(c + 3.0 * r * view / np.linalg.norm(view), c, side, side, 44.0).float())
        m = left // len(ends) + (k < left % len(ends))
        x, y, z = _cells(scene["assets"][i])[torch.randint(_cells(scene["assets"][i]).shape[0], (m,), device="cuda",
                                                           generator=gen)].unbind(1)
        u = torch.rand((m, 6), device="cuda", generator=gen, dtype=torch.float64)
        axis = (u[:, 0] * 3).long().clamp_max(2)
        face = torch.nn.functional.one_hot(axis, 3).double()
        tan1 = torch.nn.functional.one_hot((axis + 1) % 3, 3).double()
        tan2 = torch.nn.functional.one_hot((axis + 2) % 3, 3).double()
        inside = face * (u[:, 1:2] > 0.5) + tan1 * (0.1 + 0.8 * u[:, 2:3]) + tan2 * (0.1 + 0.8 * u[:, 3:4])
        p = (torch.stack([x, y, z], 1) + inside) / (1 << depth)
        phi, tilt = 2 * math.pi * u[:, 4:5], (2 * u[:, 5:6] - 1) * 1e-3
        d = tan1 * phi.cos() + tan2 * phi.sin() + face * tilt
        wt = torch.tensor(w, device="cuda")
        rays = torch.zeros((m, 8), device="cuda")
        rays[:, :3] = (p - d * (100.0 / (1 << depth))) @ wt[:3, :3].T + wt[:3, 3]
        d = d @ wt[:3, :3].T
        rays[:, 4:7] = d / d.norm(dim=1, keepdim=True)
        rays[:, 7] = math.inf
        out.append(rays)
    return torch.cat(out).contiguous()


def _request_sizes(case) -> list:
    return [REQUEST_SIZES[i % len(REQUEST_SIZES)] for i in range(case["requests"])]


def _inputs(case, seed: int) -> list:
    """The scenes of a case with their rays (and cameras), made from the seed alone."""
    rng = np.random.default_rng(seed)
    gen = torch.Generator(device="cuda").manual_seed(seed)
    kind = case["kind"]
    if kind in ("frame", "static_camera", "shaded", "host"):
        most = {11: 2, 10: 4}.get(case["depth"], 8)
        sc = _figure(rng, [(case["depth"], int(rng.integers(most))) for _ in range(case["parts"])], branch=8)
        sc["rays"] = _pinhole(*_camera(rng, sc, 1.9), case["width"], case["height"]).float()
        if kind == "static_camera":
            sc["next"] = sc["local"].copy()
            for i in range(case["parts"] - case["moving"], case["parts"]):
                a = sc["local"][i].reshape(3, 4)
                sc["next"][i] = _row(a[:, :3] @ _swing(rng.standard_normal(3), 0.1), a[:, 3])
        return [sc]
    if kind in ("graph", "served"):
        sizes = _request_sizes(case) if kind == "served" else [(case["width"], case["height"])] * case["scenes"]
        out = []
        for w, h in sizes:
            P = int(rng.integers(max(1, case["parts"] // 8), case["parts"] + 1))
            depths = rng.integers(8, 12, P)
            sc = _figure(rng, [(int(d), int(rng.integers(2 if d == 11 else 4))) for d in depths])
            sc["eye"], sc["target"] = _camera(rng, sc)
            sc["rays"], sc["size"] = _pinhole(sc["eye"], sc["target"], w, h).float(), (w, h)
            out.append(sc)
        return out
    if kind == "batch":
        size = np.exp(2 * rng.uniform(math.log(64), math.log(1024), case["scenes"]))
        n = np.maximum((size / size.sum() * case["rays"]).astype(np.int64), 1)
        n[int(n.argmax())] += case["rays"] - int(n.sum())
        out = []
        for k in range(case["scenes"]):
            sc = _cloud(rng, int(round(math.exp(rng.uniform(math.log(4), math.log(case["parts"]))))))
            sc["rays"] = _incoherent(int(n[k]), sc["box"], gen)
            out.append(sc)
        return out
    if kind == "precision":
        sc = _chains(rng, case["chains"])
        sc["rays"] = _close_up(rng, gen, sc, case["rays"])
        return [sc]
    sc = _cloud(rng, case["parts"])
    if kind == "crowd_camera":
        sc["rays"] = _pinhole(*_camera(rng, sc, 1.3), case["width"], case["height"]).float()
    else:
        sc["rays"] = _incoherent(case["rays"], sc["box"], gen)
    return [sc]


# -------------------------------------------------------------- the calls


class _State(dict):
    """What a program holds between calls; its scenes go back to the library with it."""

    def __del__(self):
        for sc in self.get("scenes", ()):
            sc.close()


def prepare(case, seed: int) -> dict:
    ctx, kind = _context(), case["kind"]
    made = _inputs(case, seed)
    scenes = [ctx.scene([_handle(a) for a in sc["assets"]], sc["parent"]) for sc in made]
    for s, sc in zip(scenes, made):
        s.set_transforms(sc["local"])
        s.refit()
    n = [sc["rays"].shape[0] for sc in made]
    rays = torch.cat([sc["rays"] for sc in made]) if len(made) > 1 else made[0]["rays"]
    hits = torch.zeros((sum(n), 2), dtype=torch.int64, device="cuda")
    state = _State(kind=kind, ctx=ctx, scenes=scenes, local=[sc["local"] for sc in made], rays=rays, hits=hits)
    state["flags"] = svo.TRACE_DEFAULT
    if kind in ("frame", "static_camera", "shaded", "host", "crowd_camera"):
        state["flags"] |= svo.trace_image(case["width"])
    if case.get("plain"):
        state["flags"] &= ~(svo.TRACE_CULL | svo.TRACE_SORT)
    state["flags"] |= {"crowd_camera": svo.TRACE_GRID, "crowd_inside": svo.TRACE_WAVEFRONT,
                       "batch": svo.TRACE_WAVEFRONT, "ordered": svo.TRACE_ORDER_ORIGIN}.get(kind, 0)
    if len(made) > 1 or kind in ("graph", "served", "batch"):
        at = np.cumsum([0] + n)
        width = [sc["size"][0] if "size" in sc else 0 for sc in made]
        state["views"] = [(rays[a:b], hits[a:b]) for a, b in zip(at[:-1], at[1:])]
        state["items"] = [(s, r, h, None, w) for s, (r, h), w in zip(scenes, state["views"], width)]
    if kind == "static_camera":
        state["poses"], state["frame"] = [made[0]["local"], made[0]["next"]], 0
        scenes[0].trace(rays, hits, flags=state["flags"])  # the frame before: its hits are kept
    elif kind == "graph":
        state["graph"] = BatchGraph(ctx, state["items"], state["local"], flags=state["flags"])
    elif kind == "served":
        state["requests"] = [(tuple(sc["eye"]), tuple(sc["target"]), *sc["size"]) for sc in made]
    elif kind == "batch":
        state["local"] = [torch.from_numpy(m).cuda() for m in state["local"]]
    elif kind == "host":
        state["rays"] = rays.cpu().pin_memory()
        state["hits"] = torch.zeros((n[0], 2), dtype=torch.int64).pin_memory()
    return state


def run(state) -> dict:
    kind, hits, rays, flags, ctx = (state[k] for k in ("kind", "hits", "rays", "flags", "ctx"))
    scene, out = state["scenes"][0], {}
    if kind == "graph":
        state["graph"].replay(state["local"])
        torch.cuda.current_stream().wait_stream(state["graph"].stream)
    elif kind == "batch":
        ctx.refit_batch(state["scenes"], state["local"])
        ctx.trace_batch(state["items"], flags=flags)
    elif kind == "served":
        for s, local in zip(state["scenes"], state["local"]):
            s.set_transforms(local)
        ctx.refit_batch(state["scenes"])
        for (eye, target, w, h), (r, _) in zip(state["requests"], state["views"]):
            ctx.raygen(eye, target, w, h, rays=r)
        ctx.trace_batch(state["items"], flags=flags)
        out["rays"] = rays
    elif kind == "static_camera":
        state["frame"] += 1
        scene.set_transforms(state["poses"][state["frame"] % 2])
        scene.refit()
        scene.trace(rays, hits, flags=flags | svo.TRACE_REUSE)
    else:
        scene.set_transforms(state["local"][0])
        scene.refit()
        if kind == "host":
            scene.trace_host(rays, hits, flags=flags)
        else:
            scene.trace(rays, hits, flags=flags)
        if kind == "shaded":
            out["colors"] = scene.hit_colors(hits)
            out["image"] = scene.shade(rays, hits, (0.3, 0.8, 0.5))
    out["t"] = hits.view(torch.float32)[:, 0]
    out["part"] = hits.view(torch.int32)[:, 1]
    out["voxel"] = hits[:, 1]
    return out


# ------------------------------------------------- the same in 64 bits


def _cells(asset) -> torch.Tensor:
    """Integer coordinates of a model's leaves."""
    key = ("cells", asset)
    if key not in _library:
        depth, ids = asset[0], _leaf_ids(*asset)
        m = (1 << depth) - 1
        _library[key] = torch.stack([ids & m, (ids >> depth) & m, ids >> (2 * depth)], 1)
    return _library[key]


def _levels(asset) -> list:
    """Sorted keys x | y << 21 | z << 42 of the occupied cells of every level below the root."""
    key = ("levels", asset)
    if key not in _library:
        c, out = _cells(asset), []
        for _ in range(asset[0]):
            out.insert(0, (c[:, 0] | (c[:, 1] << 21) | (c[:, 2] << 42)).unique())
            k = out[0] & 0x1FFFFF, (out[0] >> 21) & 0x1FFFFF, out[0] >> 42
            c = torch.stack(k, 1) >> 1
        _library[key] = out
    return _library[key]


def _closest(scene, rays) -> torch.Tensor:
    """t of the closest leaf of each ray: every occupied cell the segment meets, level by level, in 64 bits."""
    rays = rays.double()
    tmin, tmax = rays[:, 3], rays[:, 7]
    best = torch.full_like(tmin, math.inf)
    inv = np.linalg.inv(_compose(scene["local"], scene["parent"]))
    step = torch.tensor([[k & 1, (k >> 1) & 1, k >> 2] for k in range(8)], device="cuda")

    def slab(o, d, lo, size, t0, t1):
        a, b = (lo - o) / d, (lo + size - o) / d
        flat = d == 0
        if bool(flat.any()):
            inside = (o >= lo) & (o <= lo + size)
            a = torch.where(flat, torch.where(inside, -math.inf, math.inf), a)
            b = torch.where(flat, torch.where(inside, math.inf, math.inf), b)
        t0 = torch.maximum(t0, torch.minimum(a, b).amax(-1))
        return t0, torch.minimum(t1, torch.maximum(a, b).amin(-1))

    for p, asset in enumerate(scene["assets"]):
        if asset is None:
            continue
        m = torch.tensor(inv[p], device="cuda")
        # only rays that meet the sphere around the unit cube go on (1% wider than the cube needs)
        w = np.linalg.inv(inv[p])
        c = torch.tensor(w[:3, :3] @ np.full(3, 0.5) + w[:3, 3], device="cuda")
        reach = 1.01 * max(np.linalg.norm(w[:3, :3] @ (np.array(k) - 0.5)) for k in np.ndindex(2, 2, 2))
        l = c - rays[:, :3]
        dd = (rays[:, 4:7] ** 2).sum(1)
        tc = (l * rays[:, 4:7]).sum(1) / dd
        near = ((l - tc[:, None] * rays[:, 4:7]) ** 2).sum(1) <= reach * reach
        r = torch.nonzero(near & (tc + reach / dd.sqrt() >= tmin)).reshape(-1)
        o, d = rays[r, :3] @ m[:3, :3].T + m[:3, 3], rays[r, 4:7] @ m[:3, :3].T
        t0, t1 = slab(o, d, torch.zeros((), device="cuda", dtype=torch.float64), 1.0, tmin[r], tmax[r])
        k = torch.nonzero((t0 <= t1) & (t0 <= best[r])).reshape(-1)
        o, d, r = o[k], d[k], r[k]
        at = torch.arange(r.numel(), device="cuda")  # frontier: the ray and the cell of every node it meets
        cell = torch.zeros((r.numel(), 3), dtype=torch.int64, device="cuda")
        for level, keys in enumerate(_levels(asset)):
            if not at.numel():
                break
            child = 2 * cell[:, None, :] + step
            key = (child[..., 0] | (child[..., 1] << 21) | (child[..., 2] << 42)).reshape(-1)
            pos = torch.searchsorted(keys, key).clamp_max(keys.numel() - 1)
            here = torch.nonzero(keys[pos] == key).reshape(-1)
            at, cell = at[here // 8], child.reshape(-1, 3)[here]
            size = 0.5 ** (level + 1)
            t0, t1 = slab(o[at], d[at], cell.double() * size, size, tmin[r[at]], tmax[r[at]])
            k = torch.nonzero((t0 <= t1) & (t0 <= best[r[at]])).reshape(-1)
            at, cell, t0 = at[k], cell[k], t0[k]
        if at.numel():
            best.scatter_reduce_(0, r[at], t0, "amin")
    return best


def exact(case, seed: int):
    made = _inputs(case, seed)
    out = {"t": None, "part": None, "voxel": None}
    if case["kind"] == "served":
        # the rays are an output here; a hit's t follows their 32-bit values, so it has no value of its own
        out["rays"] = torch.cat([_pinhole(sc["eye"], sc["target"], *sc["size"]) for sc in made])
        return out
    if case["kind"] == "shaded":
        out["colors"] = out["image"] = None
    for sc in made:
        if "next" in sc:
            sc["local"] = sc["next"]
    out["t"] = torch.cat([_closest(sc, sc["rays"]) for sc in made])
    return out
