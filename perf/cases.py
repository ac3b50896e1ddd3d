"""The work a user of this library has it do, as cases that can be timed one by one: closest-hit
ray casting on device and host buffers, the hash-grid build, progressive photon mapping in each of
its modes, the gradient of a render, and many scenes per launch.

Sizes are those of the repository's configurations and tests, ragged variants of them among them.
A case's geometry is part of the case; its rays, points, materials and random streams come from
the seed.
"""
from __future__ import annotations

import dataclasses
import functools
import math

import numpy as np
import torch

from paper_1505_06022_gb300 import gsp, inputs as I


def listed():
    return [
        # a query of a few rays (picking, a probe, one step of an interactive tool): latency counts
        dict(name="trace_1k", kind="trace", scene="sphere", size=40, rays=1021, mix="random", uv=False,
             method="mtbvh", builder="host"),
        # an incoherent batch with barycentrics, as a user's own path tracer would send it, on a
        # mid-sized scene; a ragged count
        dict(name="trace_262k_uv", kind="trace", scene="full", size=256, rays=262147, mix="random", uv=True,
             method="mtbvh", builder="host"),
        # the closest-hit benchmark: 1,003,520 triangles, half camera rays, half random rays
        dict(name="trace_4m", kind="trace", scene="sphere", size=224, rays=4194304, mix="both", uv=False,
             method="mtbvh", builder="host"),
        # rays and results in pinned host memory
        dict(name="trace_host_1m", kind="trace_host", scene="full", size=256, rays=1048576, mix="both", uv=False),
        # the exact grid as an operation of its own, at its test's largest size
        dict(name="grid_1m", kind="grid", n=1000003, log2_table=21, cell=0.004),
        # the smallest configuration: Cornell box, a short progressive render
        dict(name="cornell_64", kind="sppm", scene="cornell", size=0, w=64, h=64, photons=16384, passes=4,
             r0_frac=0.05, photon_mode=gsp.FULL_PATH, hash_mode=gsp.EXACT),
        # one pass at a time at a ragged preview size: no other pass to overlap with
        dict(name="preview_131x97", kind="sppm", scene="full", size=64, w=131, h=97, photons=65536, passes=1,
             r0_frac=0.004, photon_mode=gsp.FULL_PATH, hash_mode=gsp.EXACT),
        # the large render: 247,234 triangles with glass and mirror, 512 x 512, 2^20 photon paths
        dict(name="sppm_512", kind="sppm", scene="full", size=256, w=512, h=512, photons=1 << 20, passes=8,
             r0_frac=0.004, photon_mode=gsp.FULL_PATH, hash_mode=gsp.EXACT),
        # smooth normals and textures, ragged image and photon count
        dict(name="shaded_333x217", kind="sppm", scene="shaded", size=256, w=333, h=217, photons=262147, passes=4,
             r0_frac=0.004, photon_mode=gsp.FULL_PATH, hash_mode=gsp.EXACT),
        # the paper's own photon pass: one bounce per pass, stochastic hashing
        dict(name="regen_stoch_256", kind="sppm", scene="full", size=256, w=256, h=256, photons=1 << 18, passes=4,
             r0_frac=0.004, photon_mode=gsp.REGEN, hash_mode=gsp.STOCHASTIC),
        # one step of a material fit: forward render, loss, gradient by path replay
        dict(name="fit_256", kind="fit", scene="grad", size=128, w=256, h=256, photons=1 << 18, passes=8,
             r0_frac=0.004),
        # uneven scenes rendered together as one graph
        dict(name="batch_16", kind="batch", scenes=16, photons=1 << 18, passes=2, r0_frac=0.004),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["trace", "trace", "trace_host", "grid", "sppm", "sppm", "sppm", "grad", "fit", "batch"])
    if kind in ("trace", "trace_host"):
        scene = rng.choice(["sphere", "full", "soup"])
        size = {"sphere": lambda: _log(rng, 8, 224), "full": lambda: _log(rng, 16, 256),
                "soup": lambda: _log(rng, 100, 3000)}[scene]()
        case = dict(kind=kind, scene=scene, size=size, rays=_log(rng, 1, 4_000_000 if kind == "trace" else 1_000_000),
                    mix=rng.choice(["camera", "random", "both"]), uv=rng.random() < 0.4)
        if kind == "trace":
            case["builder"] = rng.choice(["host", "host", "device"])
            case["method"] = rng.choice(["mtbvh", "mtbvh", "mtbvh", "stack"])
        return case
    if kind == "grid":
        n = _log(rng, 100, 1_000_000)
        return dict(kind=kind, n=n, log2_table=min(21, max(6, n.bit_length() + rng.choice([0, 1]))),
                    cell=rng.choice([0.004, 0.01, 0.05]))
    if kind == "sppm":
        scene = rng.choice(["cornell", "full", "full", "shaded", "grad"])
        return dict(kind=kind, scene=scene, size=0 if scene == "cornell" else _log(rng, 24, 256),
                    w=_log(rng, 48, 500), h=_log(rng, 48, 500), photons=_log(rng, 4000, 700_000),
                    passes=rng.choice([1, 2, 3, 5]), r0_frac=rng.choice([0.004, 0.008]) if scene != "cornell" else 0.05,
                    photon_mode=rng.choice([gsp.FULL_PATH, gsp.FULL_PATH, gsp.REGEN]),
                    hash_mode=rng.choice([gsp.EXACT, gsp.EXACT, gsp.STOCHASTIC]))
    if kind in ("grad", "fit"):
        return dict(kind=kind, scene="grad", size=_log(rng, 24, 128), w=_log(rng, 48, 256), h=_log(rng, 48, 256),
                    photons=_log(rng, 4000, 262_144), passes=rng.choice([1, 2, 4, 8]), r0_frac=0.004)
    return dict(kind=kind, scenes=rng.choice([2, 3, 5, 8, 11]), photons=_log(rng, 16_000, 262_144),
                passes=rng.choice([1, 2, 3]), r0_frac=0.004)


# ---- inputs ------------------------------------------------------------------------------------
@functools.lru_cache(maxsize=4)
def _geometry(scene, size, w, h):
    if scene == "sphere":
        return I.traversal_sphere(n=size, seed=2)
    if scene == "soup":
        return I.random_soup(size, seed=31, size=0.15)
    if scene == "cornell":
        return I.cornell_box(seed=1, width=w, height=h)
    if scene == "grad":
        return I.grad_scene(seed=4, width=w, height=h, plane_quads=size, sphere_n=max(2, size * 15 // 128))
    make = {"full": I.full_scene, "shaded": I.shaded_scene}[scene]
    return make(width=w, height=h, plane_quads=size, sphere_n=max(2, size * 44 // 256))


@functools.lru_cache(maxsize=2)
def _batch_geometry(count):
    return I.batch_scenes(count, seed=5)


def _materials(sc, seed):
    """The scene with the albedos of its diffuse materials drawn again from the seed."""
    rng = np.random.default_rng(seed)
    mats = sc.mats.copy()
    for i in range(len(mats)):
        if mats["type"][i] == I.DIFFUSE:
            mats["albedo"][i] = rng.uniform(0.2, 0.8, 3)
    return dataclasses.replace(sc, mats=mats)


def _rays(case, sc, seed):
    """[n, 8] rays on the GPU: pinhole rays in row-major order (every ray of "camera", the first
    half of "both") and rays of uniform origin and direction."""
    n = case["rays"]
    dev = torch.device("cuda")
    g = torch.Generator(device=dev)
    g.manual_seed(seed)
    lo, hi = sc.verts.min(axis=0).astype(np.float64), sc.verts.max(axis=0).astype(np.float64)
    center, half = (lo + hi) / 2, (hi - lo) / 2
    nc = {"camera": n, "random": 0, "both": n // 2}[case["mix"]]
    rays = torch.zeros((n, 8), dtype=torch.float32, device=dev)
    rays[:, 7] = float("inf")
    if nc:
        r = np.random.default_rng(seed)
        eye = r.normal(size=3) * (1.0, 0.3, 1.0)
        eye = center + eye / np.linalg.norm(eye) * 1.5 * float(np.linalg.norm(half))
        fwd = (center - eye) / np.linalg.norm(center - eye)
        right = np.cross(fwd, (0.0, 1.0, 0.0))
        right /= np.linalg.norm(right)
        up = np.cross(right, fwd)
        w = max(1, int(math.sqrt(2 * nc)))
        h = -(-nc // w)
        i = torch.arange(nc, device=dev)
        th = math.tan(math.radians(45.0) / 2)
        sx = (((i % w).double() + 0.5) / w * 2 - 1) * th * w / h
        sy = (1 - ((i // w).double() + 0.5) / h * 2) * th
        t = lambda v: torch.tensor(v, dtype=torch.float64, device=dev)  # noqa: E731
        d = t(fwd) + sx[:, None] * t(right) + sy[:, None] * t(up)
        rays[:nc, 0:3] = t(eye).float()
        rays[:nc, 4:7] = (d / d.norm(dim=1, keepdim=True)).float()
    if n > nc:
        u = torch.rand((n - nc, 3), generator=g, device=dev) * 2 - 1
        scale = torch.tensor(half * (2.0 if case["scene"] == "sphere" else 1.2), dtype=torch.float32, device=dev)
        rays[nc:, 0:3] = torch.tensor(center, dtype=torch.float32, device=dev) + u * scale
        d = torch.randn((n - nc, 3), generator=g, device=dev)
        rays[nc:, 4:7] = d / d.norm(dim=1, keepdim=True)
    return rays


def _params(case, sc, seed, scene_id=0):
    return gsp.sppm_params(sc, case["photons"], seed=seed, r0_frac=case["r0_frac"],
                           photon_mode=case.get("photon_mode", gsp.FULL_PATH),
                           hash_mode=case.get("hash_mode", gsp.EXACT), scene_id=scene_id)


def prepare(case, seed):
    kind = case["kind"]
    ctx = gsp.Context(0)
    st = dict(case=case, ctx=ctx)
    if kind in ("trace", "trace_host"):
        sc = _geometry(case["scene"], case["size"], 64, 64)
        rays = _rays(case, sc, seed)
        if kind == "trace":
            st.update(scene=gsp.Scene(ctx, sc, builder=case["builder"]), rays=rays)
        else:
            n = case["rays"]
            pin = lambda *shape, dtype: torch.empty(shape, dtype=dtype, pin_memory=True)  # noqa: E731
            st.update(scene=gsp.Scene(ctx, sc), rays=rays.cpu().pin_memory(), tri=pin(n, dtype=torch.int32),
                      t=pin(n, dtype=torch.float32), uv=pin(n, 2, dtype=torch.float32) if case["uv"] else None)
        return st
    if kind == "grid":
        n = case["n"]
        g = torch.Generator(device="cuda")
        g.manual_seed(seed)
        pos = torch.zeros((n, 4), dtype=torch.float32, device="cuda")
        pos[:, :3] = torch.randn((n, 3), generator=g, device="cuda")
        pos[: n // 2, :3] *= 1.5   # a diffuse cloud
        pos[n // 2:, :3] *= 0.02   # a dense clump, as under a caustic
        st.update(pos=pos)
        return st
    if kind == "batch":
        rs = []
        for i, sc in enumerate(_batch_geometry(case["scenes"])):
            sc = _materials(sc, 1000 * seed + i)
            rs.append(gsp.Renderer(gsp.Scene(ctx, sc), _params(case, sc, seed + i, scene_id=i)))
        st.update(renderers=rs, batch=gsp.Batch(rs))
        return st
    sc = _materials(_geometry(case["scene"], case["size"], case["w"], case["h"]), seed)
    scene = gsp.Scene(ctx, sc)
    params = _params(case, sc, seed)
    st.update(scene=scene)
    if kind == "sppm":
        st.update(renderer=gsp.Renderer(scene, params))
        return st
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    if kind == "grad":  # the forward passes are done; run() is their gradient
        r = gsp.Renderer(scene, params)
        r.enable_grad(case["passes"])
        r.run(case["passes"])
        img = r.image()
        st.update(renderer=r, dloss=img * (torch.rand(img.shape, generator=g, device="cuda") - 0.5))
        return st
    # fit: the target is a render at other albedos
    em = gsp.emitting_material(sc.mats)
    albedo = torch.tensor(sc.mats["albedo"], device="cuda")
    emission = torch.tensor(sc.mats["emission"][em], device="cuda")
    factor = 0.8 + 0.4 * torch.rand(albedo.shape, generator=g, device="cuda")
    with torch.no_grad():
        target = gsp.render((albedo * factor).clamp(0.0, 0.95), emission, scene, params, case["passes"])
    st.update(params=params, target=target.detach(), albedo=albedo.requires_grad_(),
              emission=emission.requires_grad_())
    return st


def _progress(r):
    s = r.state()
    return {"image": r.image(), "N": s["N"], "R": s["R"], "tau": s["tau"], "direct": s["direct"]}


def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "trace":
        out = st["scene"].trace(st["rays"], with_uv=case["uv"], method=case["method"])
        return dict(zip(("tri", "t", "uv"), out))
    if kind == "trace_host":
        gsp.gsp_trace_closest_hit_host(st["scene"].h, st["rays"], st["tri"], st["t"], st["uv"])
        return {"tri": st["tri"], "t": st["t"], "uv": st["uv"]}
    if kind == "grid":
        order, start = gsp.gsp_hash_grid_build(st["ctx"].h, st["pos"], case["cell"], 1 << case["log2_table"])
        return {"order": order, "start": start}
    if kind == "sppm":
        st["renderer"].run(case["passes"])
        return _progress(st["renderer"])
    if kind == "batch":
        st["batch"].run(case["passes"])
        return [{"image": r.image(), "state": r.state()["tau"]} for r in st["renderers"]]
    if kind == "grad":
        albedo, emission = st["renderer"].grad(st["dloss"])
        return {"albedo": albedo, "emission": emission}
    for p in (st["albedo"], st["emission"]):
        p.grad = None
    img = gsp.render(st["albedo"], st["emission"], st["scene"], st["params"], case["passes"])
    loss = 0.5 * (img - st["target"]).square().sum()
    loss.backward()
    return {"image": img.detach(), "loss": loss.detach(), "albedo": st["albedo"].grad, "emission": st["emission"].grad}


# ---- what a pass cannot do without -------------------------------------------------------------
def _triangles(scene, size):
    return {"sphere": 20 * size * size, "soup": size, "cornell": 36,
            "grad": 2 * size * size + 80 * max(2, size * 15 // 128) ** 2 + 2}.get(
                scene, 2 * size * size + 60 * max(2, size * 44 // 256) ** 2 + 2)


def _ray_flops(nt):
    """A descent of a binary tree over nt triangles (12 operations per box) and one triangle test."""
    return 12 * math.log2(max(2, nt)) + 30


def _render_work(nt, npix, photons, passes):
    """Triangles (36 bytes) read once; per pass the pixel state (32 bytes) read and written and, for
    about half of the photon paths, a deposit (32 bytes) written and read. One eye ray per pixel and
    about 1.5 rays per photon path."""
    return {"bytes": 36 * nt + passes * (64 * npix + 0.5 * 64 * photons),
            "flops": passes * (npix + 1.5 * photons) * _ray_flops(nt)}


def work(case):
    kind = case["kind"]
    if kind in ("trace", "trace_host"):
        nt, n = _triangles(case["scene"], case["size"]), case["rays"]
        # a batch of fewer rays than triangles touches one triangle per ray
        return {"bytes": n * (40 + (8 if case["uv"] else 0)) + 36 * min(n, nt), "flops": n * _ray_flops(nt)}
    if kind == "grid":
        return {"bytes": 20 * case["n"] + 4 * (1 << case["log2_table"]), "flops": 20 * case["n"]}
    if kind == "batch":
        parts = [_render_work(sc.ntris, int(sc.camera["width"][0]) * int(sc.camera["height"][0]), case["photons"],
                              case["passes"]) for sc in _batch_geometry(case["scenes"])]
        return {k: sum(p[k] for p in parts) for k in ("bytes", "flops")}
    w = _render_work(_triangles(case["scene"], case["size"]), case["w"] * case["h"], case["photons"], case["passes"])
    if kind == "fit":  # the gradient replays the paths of the forward passes
        return {k: 2 * v for k, v in w.items()}
    return w


# ---- the same in 64 bits -----------------------------------------------------------------------
def exact(case, seed):
    """Hit distances of a query over few triangles by brute force in FP64; the renders have no such
    value (their estimate is defined by the library's random streams)."""
    if case["kind"] not in ("trace", "trace_host"):
        return None
    n, nt = case["rays"], _triangles(case["scene"], case["size"])
    if n * nt > 1_000_000_000:
        return None
    sc = _geometry(case["scene"], case["size"], 64, 64)
    rays = _rays(case, sc, seed).double()
    v = torch.from_numpy(sc.verts).cuda().double()[torch.from_numpy(sc.tris).cuda().long()]
    v0, e1, e2 = v[:, 0], v[:, 1] - v[:, 0], v[:, 2] - v[:, 0]
    out = torch.empty(n, dtype=torch.float64, device="cuda")
    step = max(1, 30_000_000 // nt)
    for a in range(0, n, step):
        o, d = rays[a:a + step, None, 0:3], rays[a:a + step, None, 4:7]
        p = torch.linalg.cross(d.expand(-1, nt, -1), e2[None].expand(d.shape[0], -1, -1))
        det = (e1[None] * p).sum(-1)
        s = o - v0[None]
        u = (s * p).sum(-1) / det
        del p
        q = torch.linalg.cross(s, e1[None].expand(s.shape[0], -1, -1))
        w = (d * q).sum(-1) / det
        t = (e2[None] * q).sum(-1) / det
        ok = (det != 0) & (u >= 0) & (w >= 0) & (u + w <= 1) & (t > rays[a:a + step, None, 3])
        out[a:a + step] = torch.where(ok, t, float("inf")).min(dim=1).values
    t = out if case["kind"] == "trace" else out.cpu()
    return {"tri": None, "t": t, "uv": None}
