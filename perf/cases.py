"""Workloads this library is timed on, through its public Python entry points.

Each case stands for a call a program makes in earnest: whole octree builds from
the smallest clouds to the largest, a batch of clouds, the previews, the digest
that keys the build cache, a rendered frame and an out-of-core build.  Clouds are
made on the GPU from a seed: points uniform in a cube, or a scanner scene (a few
scanners on wavy ground among boxes, density falling with the distance squared),
in random order or scan after scan as a file of merged scans holds them.
"""
import math

import numpy as np
import torch

from paper_2302_05002_gb300 import fastpoints as fp

BLOCK = 1 << 24   # points generated at a time


# ------------------------------------------------------------------ the cases
def listed():
    return [
        # a small scan, parameters of the smoke build: latency and launches count
        dict(name="build-20k", path="build", api="octree", cloud="lidar", order="random", n=20_000, sub=7, lmax=15,
             T=2_000, C=500),
        # the 1M uniform workload through the convenience call, leaf-grouped points included
        dict(name="build-1m", path="build", api="octree", cloud="uniform", order="random", n=1_000_000, sub=7,
             lmax=15, T=100_000, C=20_000),
        # a cloud as a serving process builds it: the plain calls on kept buffers, points scan after scan
        dict(name="build-10m-scans", path="build", api="plain", cloud="lidar", order="scans", n=9_999_991, sub=7,
             lmax=15, T=100_000, C=20_000),
        # the 100M LiDAR workload as the benchmark runs it (the count's cells handed to the distribution)
        dict(name="build-100m", path="build", api="cells", cloud="lidar", order="random", n=100_000_000, sub=7,
             lmax=15, T=100_000, C=20_000),
        # the parameters of the 10^9-point workload at half its points
        dict(name="build-500m", path="build", api="cells", cloud="uniform", order="random", n=500_000_000, sub=7,
             lmax=8, T=5_000_000, C=50_000),
        # many clouds in one call: sizes log-uniform, uniform or LiDAR by a coin flip
        dict(name="batch-48", path="batch", count=48, lo=10_000, hi=4_000_000, fused=True, lanes=32),
        # one streamed piece of a served cloud: the preview of 8M points with its place in the cloud
        dict(name="piece-8m", path="decimate", cloud="lidar", n=1 << 23, first=3 << 23, modulus=16),
        # preview and extent of a cloud under a budget of about 10^6 points (modulus no power of two)
        dict(name="preview-51m", path="preview", cloud="lidar", n=51_161_407, modulus=52),
        # the spatially even preview of a large scan: one point per occupied cell
        dict(name="spatial-100m", path="spatial", cloud="lidar", order="random", n=100_000_000, level=7),
        # the digest that looks a cloud up in the build cache
        dict(name="digest-30m", path="digest", cloud="uniform", n=29_999_999),
        # one frame of a resident octree at 1920 x 1080
        dict(name="render-30m", path="render", cloud="lidar", n=30_000_000, width=1920, height=1080, px=30.0),
        # a cloud in pinned host memory built inside a device arena, in streamed pieces
        dict(name="out-of-core-12m", path="ooc", cloud="lidar", n=12_000_007, piece=1 << 21),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    path = rng.choice(["build"] * 6 + ["batch", "decimate", "preview", "spatial", "digest", "render", "ooc"])
    cloud = rng.choice(["uniform", "lidar"])
    if path == "build":
        # uniform clouds of every size; a scene costs more per point and stays below 200M
        n = _log(rng, 5_000, 400_000_000 if cloud == "uniform" else 150_000_000)
        C = min(50_000, max(100, _log(rng, n / 4_000 + 50, n / 40 + 100)))
        T = min(5_000_000, max(C, _log(rng, C, 10 * C)))
        return dict(path=path, api=rng.choice(["octree", "plain", "cells"]), cloud=cloud,
                    order=rng.choice(["random", "scans"]), n=n, sub=7, lmax=rng.choice([8, 10, 12, 15]), T=T, C=C)
    if path == "batch":
        return dict(path=path, count=rng.randint(4, 64), lo=10_000, hi=_log(rng, 100_000, 4_000_000),
                    fused=rng.random() < 0.5, lanes=rng.choice([4, 8, 16, 32]))
    if path == "decimate":
        return dict(path=path, cloud=cloud, n=_log(rng, 10_000, 1 << 23), first=rng.randrange(1 << 30),
                    modulus=rng.choice([4, 16, 100]))
    if path == "preview":
        n = _log(rng, 100_000, 400_000_000)
        return dict(path=path, cloud=cloud, n=n, modulus=rng.choice([16, max(1, -(-n // 1_000_000))]))
    if path == "spatial":
        return dict(path=path, cloud=cloud, order=rng.choice(["random", "scans"]), n=_log(rng, 100_000, 200_000_000),
                    level=rng.randint(5, 7))
    if path == "digest":
        return dict(path=path, cloud=cloud, n=_log(rng, 10_000, 200_000_000))
    if path == "render":
        w, h = rng.choice([(1280, 720), (1920, 1080), (3840, 2160), (801, 599)])
        return dict(path=path, cloud=cloud, n=_log(rng, 500_000, 60_000_000), width=w, height=h,
                    px=rng.choice([10.0, 30.0, 100.0]))
    return dict(path=path, cloud=cloud, n=_log(rng, 500_000, 16_000_000), piece=1 << rng.randint(19, 22))


def _params(case):
    return fp.params(grid_log2=7, sub_log2=case.get("sub", 7), max_level=case.get("lmax", 15),
                     decim_modulus=case.get("modulus", 16), chunk_threshold=case.get("T", 100_000),
                     node_capacity=case.get("C", 20_000))


# ------------------------------------------------------------------ the clouds
def _scene(seed):
    """Scanners, boxes and ground waves of one scene (mm; 500 m x 500 m x 60 m)."""
    r = np.random.default_rng(seed)
    scan = r.uniform(0.0, 500_000.0, (40, 2))
    size = r.uniform([5_000, 5_000, 4_000], [40_000, 40_000, 40_000], (200, 3))
    low = r.uniform(0.0, 1.0, (200, 2)) * (500_000.0 - size[:, :2])
    wave = r.uniform(0.0, 2 * math.pi, (4, 2))
    return scan, np.concatenate([low, size], 1), wave


def _ground(x, y, wave):
    z = torch.full_like(x, 8_000.0)
    for k, (a, b) in enumerate(wave.tolist()):
        f = 2 * math.pi / (250_000.0 / (k + 1))
        z += 1_800.0 / (k + 1) * (torch.sin(x * f + a) + torch.sin(y * f + b))
    return z


def _lidar_block(at, n, total, order, scene, gen):
    dev = "cuda"
    scan, box, wave = scene
    u = lambda: torch.rand(n, device=dev, generator=gen)   # noqa: E731
    if order == "scans":   # scan after scan, each one turn of its scanner
        pos = torch.arange(at, at + n, device=dev, dtype=torch.float64) * (40.0 / total)
        s = pos.floor().clamp_(0, 39).to(torch.int64)
        turn = (pos - s).to(torch.float32)
    else:
        s = torch.randint(0, 40, (n,), device=dev, generator=gen)
        turn = u()
    sc = torch.as_tensor(scan, dtype=torch.float32, device=dev)[s]
    # ground: radius with density rho / (rho^2 + h^2) up to 250 m, from 1.8 m above it
    h = 1_800.0
    rho = h * torch.sqrt(torch.exp(u() * math.log(1.0 + (250_000.0 / h) ** 2)) - 1.0)
    x, y = sc[:, 0] + rho * torch.cos(2 * math.pi * turn), sc[:, 1] + rho * torch.sin(2 * math.pi * turn)
    x, y = x.abs(), y.abs()
    x, y = torch.where(x > 499_999.0, 999_998.0 - x, x), torch.where(y > 499_999.0, 999_998.0 - y, y)
    z = _ground(x, y, wave)
    # a third of the returns from walls and roofs of the boxes
    bx = torch.as_tensor(box, dtype=torch.float32, device=dev)[torch.randint(0, 200, (n,), device=dev, generator=gen)]
    face, a, b = torch.randint(0, 5, (n,), device=dev, generator=gen), u(), u()
    wx = torch.where(face == 2, torch.zeros_like(a), torch.where(face == 3, torch.ones_like(a), a))
    wy = torch.where(face == 0, torch.zeros_like(a), torch.where(face == 1, torch.ones_like(a),
                                                                torch.where(face == 4, b, a)))
    wz = torch.where(face == 4, torch.ones_like(b), b)
    wall = u() < 0.33
    x = torch.where(wall, bx[:, 0] + wx * bx[:, 2], x)
    y = torch.where(wall, bx[:, 1] + wy * bx[:, 3], y)
    z = torch.where(wall, 8_000.0 + wz * bx[:, 4], z)
    p = torch.stack([x, y, z], 1)
    del x, y, z, wx, wy, wz, bx
    p += 5.0 * torch.randn((n, 3), device=dev, generator=gen)
    top = torch.tensor([499_999.0, 499_999.0, 59_999.0], device=dev)
    out = torch.empty((n, 4), dtype=torch.int32, device=dev)
    out[:, :3] = torch.minimum(p.round_(), top).clamp_(min=0.0).to(torch.int32)
    shade = (out[:, 2] >> 8) + torch.randint(-16, 17, (n,), device=dev, generator=gen, dtype=torch.int32)
    shade.clamp_(0, 255)
    out[:, 3] = shade | ((255 - shade) << 8) | ((shade >> 1) << 16) | -16777216
    return out


def cloud(kind, n, seed, order="random"):
    """(n, 4) int32 points on the GPU."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed))
    pts = torch.empty((n, 4), dtype=torch.int32, device="cuda")
    scene = _scene(int(seed)) if kind == "lidar" else None
    for at in range(0, n, BLOCK):
        m = min(BLOCK, n - at)
        if kind == "lidar":
            pts[at:at + m] = _lidar_block(at, m, n, order, scene, gen)
        else:
            pts[at:at + m, :3] = torch.randint(0, 1 << 20, (m, 3), device="cuda", generator=gen, dtype=torch.int32)
            pts[at:at + m, 3] = torch.randint(-(1 << 31), 1 << 31, (m,), device="cuda", generator=gen).to(torch.int32)
    return pts


# ------------------------------------------------------------------ preparing
_STAGES = ("bounds_decimate", "merge", "distribute", "octree", "subsample")


def _kept_outputs(pts, prm, leaf):
    out = fp.cloud_outputs(pts, prm, leaf=leaf)
    for t in out.values():   # what a build leaves unwritten stays zero
        if isinstance(t, torch.Tensor):
            t.zero_()
    return out


def prepare(case, seed):
    return globals()["_prepare_" + case["path"]](case, seed)


def _prepare_build(case, seed):
    pts, prm = cloud(case["cloud"], case["n"], seed, case["order"]), _params(case)
    s = dict(path="build", api=case["api"], pts=pts, prm=prm)
    if case["api"] != "octree":
        n = pts.shape[0]
        s["out"] = _kept_outputs(pts, prm, leaf=False)
        s["ws"] = torch.empty(max(fp.workspace_size(k, n, prm) for k in _STAGES), dtype=torch.uint8, device="cuda")
        if case["api"] == "plain":
            s["desc"] = fp.cloud_desc(pts, prm, s["out"])
        else:
            s["cells"] = torch.zeros(n, dtype=torch.int32, device="cuda")
    else:
        s["kept"] = _kept_count(n=case["n"], first=0, modulus=prm.decim_modulus)
    return s


def _batch_sizes(case, seed):
    r = np.random.default_rng(int(seed) + 77)
    lo, hi = math.log(case["lo"]), math.log(case["hi"])
    # the sizes spread evenly over the logarithm, so that every seed's batch is as large
    sizes = [int(math.exp(lo + (hi - lo) * (k + 0.5) / case["count"])) for k in range(case["count"])]
    kinds = ["lidar" if k else "uniform" for k in r.integers(0, 2, case["count"])]
    order = r.permutation(case["count"])
    return [sizes[k] for k in order], kinds


def _prepare_batch(case, seed):
    prm = _params(case)
    sizes, kinds = _batch_sizes(case, seed)
    clouds = [(cloud(kind, n, int(seed) * 1000 + i), prm) for i, (n, kind) in enumerate(zip(sizes, kinds))]
    # every cloud's outputs are slices of one array per output
    off = np.concatenate([[0], np.cumsum(sizes)])
    caps = [fp.node_capacity_bound(n, prm) for n in sizes]
    noff = np.concatenate([[0], np.cumsum(caps)])
    poff = np.concatenate([[0], np.cumsum([fp._preview_cap(n, prm.decim_modulus) for n in sizes])])
    i32 = dict(dtype=torch.int32, device="cuda")
    k, cells, total = len(sizes), 1 << 21, int(off[-1])
    whole = dict(cube=torch.zeros((k, 8), **i32), preview=torch.zeros((int(poff[-1]), 4), **i32),
                 preview_count=torch.zeros(k, dtype=torch.int64, device="cuda"), counts=torch.zeros((k, cells), **i32),
                 chunks=torch.zeros((k, cells, 4), **i32), num_chunks=torch.zeros(k, **i32),
                 lut=torch.zeros((k, cells), **i32), offsets=torch.zeros((k, cells + 2), dtype=torch.int64, device="cuda"),
                 dist=torch.zeros((total, 4), **i32), perm=torch.zeros(total, **i32),
                 nodes=torch.zeros((int(noff[-1]), 10), **i32), num_nodes=torch.zeros(k, **i32),
                 owner=torch.zeros(total, **i32), final=torch.zeros((total, 4), **i32),
                 final_perm=torch.zeros(total, **i32))
    outs = []
    for i in range(k):
        a, b = int(off[i]), int(off[i + 1])
        o = {name: whole[name][a:b] for name in ("dist", "perm", "owner", "final", "final_perm")}
        o.update({name: whole[name][i] for name in ("cube", "counts", "chunks", "lut", "offsets")})
        o.update({name: whole[name][i:i + 1] for name in ("preview_count", "num_chunks", "num_nodes")})
        o.update(preview=whole["preview"][int(poff[i]):int(poff[i + 1])], nodes=whole["nodes"][int(noff[i]):int(noff[i + 1])],
                 preview_cap=int(poff[i + 1] - poff[i]), node_cap=caps[i], leaf_pts=None, leaf_perm=None)
        outs.append(o)
    opts = fp.batch_opts(case["lanes"], case["fused"], 256, 1024)
    descs = fp.batch_descs(clouds, outs)
    ws = torch.empty(fp.batch_workspace_size_ex(descs, k, opts), dtype=torch.uint8, device="cuda")
    return dict(path="batch", clouds=clouds, whole=whole, outs=outs, opts=opts, descs=descs, ws=ws)


def _prepare_decimate(case, seed):
    n = case["n"]
    return dict(path="decimate", pts=cloud(case["cloud"], n, seed), first=case["first"], modulus=case["modulus"],
                out=torch.zeros((fp._preview_cap(n, case["modulus"]), 4), dtype=torch.int32, device="cuda"),
                ws=torch.empty(fp.workspace_size("decimate", n), dtype=torch.uint8, device="cuda"))


def _prepare_preview(case, seed):
    n = case["n"]
    return dict(path="preview", pts=cloud(case["cloud"], n, seed), modulus=case["modulus"],
                out=torch.zeros((fp._preview_cap(n, case["modulus"]), 4), dtype=torch.int32, device="cuda"),
                ws=torch.empty(fp.workspace_size("bounds_decimate", n), dtype=torch.uint8, device="cuda"))


def _prepare_spatial(case, seed):
    n, level = case["n"], case["level"]
    pts = cloud(case["cloud"], n, seed, case["order"])
    prm = fp.params(grid_log2=level, sub_log2=level, max_level=level)
    need = max(fp.workspace_size("preview_spatial", n, prm), fp.workspace_size("bounds", n))
    return dict(path="spatial", pts=pts, level=level, ws=torch.empty(need, dtype=torch.uint8, device="cuda"),
                out=torch.zeros((min(n, 1 << (3 * level)), 4), dtype=torch.int32, device="cuda"))


def _prepare_digest(case, seed):
    return dict(path="digest", pts=cloud(case["cloud"], case["n"], seed))


def _prepare_render(case, seed):
    pts = cloud(case["cloud"], case["n"], seed)
    r = fp.build_octree(pts, _params(case))
    m = int(r["num_nodes"].item())
    lo, hi = pts[:, :3].amin(0).double().cpu().numpy(), pts[:, :3].amax(0).double().cpu().numpy()
    d = hi - lo
    eye = [lo[0] + 0.1 * d[0], lo[1] - 0.15 * d[1], lo[2] + 0.3 * max(d)]
    view = fp.view_projection(eye, lo + 0.5 * d, aspect=case["width"] / case["height"], near=1.0,
                              far=4.0 * float(max(d)) + 10.0)
    i64 = dict(dtype=torch.int64, device="cuda")
    return dict(path="render", nodes=r["nodes"][:m].contiguous(), num=r["num_nodes"], cube=r["cube"], final=r["final"],
                cam=fp.camera(view, case["width"], case["height"], case["px"]),
                fb=torch.empty((case["height"], case["width"]), **i64),
                ws=torch.empty(fp.render_workspace_size(m), dtype=torch.uint8, device="cuda"))


def _prepare_ooc(case, seed):
    prm, n = _params(case), case["n"]
    host = cloud(case["cloud"], n, seed).cpu().pin_memory()
    out = fp.ooc_outputs(n, prm)
    for t in out.values():
        if isinstance(t, torch.Tensor):
            t.zero_()
    return dict(path="ooc", host=host, prm=prm, piece=case["piece"], out=out,
                arena=torch.empty(fp.ooc_arena_min(n, prm, case["piece"]) + (64 << 20), dtype=torch.uint8, device="cuda"),
                scratch=torch.empty(fp.ooc_host_bytes(n, prm), dtype=torch.uint8).pin_memory())


# ------------------------------------------------------------------ one pass
def run(s):
    return globals()["_run_" + s["path"]](s)


def _run_build(s):
    pts, prm = s["pts"], s["prm"]
    if s["api"] == "octree":
        r = fp.build_octree(pts, prm)
        return [r["cube"], r["preview"][:s["kept"]], r["preview_count"], r["counts"], r["num_chunks"], r["lut"],
                r["dist"], r["perm"], r["nodes"], r["num_nodes"], r["leaf_pts"], r["leaf_perm"], r["owner"],
                r["final"], r["final_perm"]]
    o = s["out"]
    kept = ("preview", "preview_count", "counts", "num_chunks", "lut", "dist", "perm", "nodes", "num_nodes", "owner",
            "final", "final_perm")
    if s["api"] == "plain":
        fp.plain_calls(s["desc"], s["ws"])
        return [o[k] for k in ("cube", "chunks", "offsets") + kept]
    g, ws = prm.grid_log2, s["ws"]
    cube, prev, prev_n = fp.fp_bounds_decimate(pts, 0, prm.decim_modulus, out=o["preview"], ws=ws)
    counts, cells = fp.fp_count_cells(pts, cube, g, counts=o["counts"], cells=s["cells"])
    chunks, num, lut, offsets = fp.fp_merge_chunks(counts, g, prm.chunk_threshold, ws=ws)
    dist, perm = fp.fp_distribute_cells(pts, cells, cube, g, lut, offsets, num, out=o["dist"], perm=o["perm"], ws=ws)
    nodes, num_nodes, _, _, owner = fp.fp_build_chunk_octree(dist, perm, cube, chunks, num, offsets, counts, prm,
                                                             leaf=False, ws=ws)
    final, final_perm = fp.fp_subsample(nodes, num_nodes, dist, perm, owner, chunks, num, offsets, prm, ws=ws,
                                        final=o["final"], final_perm=o["final_perm"])
    return [cube, prev, prev_n, counts, cells, num, lut, dist, perm, nodes, num_nodes, owner, final, final_perm]


def _run_batch(s):
    fp.build_batched(s["clouds"], outs=s["outs"], ws=s["ws"], opts=s["opts"])
    return list(s["whole"].values())


def _run_decimate(s):
    return list(fp.fp_decimate(s["pts"], s["first"], s["modulus"], out=s["out"], ws=s["ws"]))


def _run_preview(s):
    return list(fp.fp_bounds_decimate(s["pts"], 0, s["modulus"], out=s["out"], ws=s["ws"]))


def _run_spatial(s):
    cube = fp.fp_bounds(s["pts"], ws=s["ws"])
    return [cube] + list(fp.fp_preview_spatial(s["pts"], cube, s["level"], out=s["out"], ws=s["ws"]))


def _run_digest(s):
    d = fp.fp_cloud_digest(s["pts"])
    return d - (1 << 64) if d >> 63 else d   # as a signed 64-bit number


def _run_render(s):
    ids, nsel, npts = fp.fp_select_nodes(s["nodes"], s["num"], s["cube"], s["cam"], ws=s["ws"])
    fb = fp.fp_rasterize(s["nodes"], ids, nsel, s["final"], s["cam"], fb=s["fb"], ws=s["ws"])
    return [nsel, npts, fb]


def _run_ooc(s):
    o = fp.build_ooc(s["host"], s["prm"], s["arena"], piece_points=s["piece"], scratch=s["scratch"], out=s["out"])
    return [o[k] for k in ("cube", "preview", "preview_count", "nodes", "num_nodes", "final", "final_perm")]


# ------------------------------------------------------------------ its work
def work(case):
    """Bytes of one pass: each input read once, each output written once."""
    path, grid = case["path"], 4 << 21
    if path == "batch":
        n, k = sum(_batch_sizes(case, 0)[0]), case["count"]
        return {"bytes": n * (16 + 1 + 20 + 4 + 20) + k * 2 * grid, "flops": 0}
    n = case["n"]
    if path == "build":
        per = 16 + 1 + 20 + 4 + 20 + {"octree": 20, "plain": 0, "cells": 4}[case["api"]]
        return {"bytes": n * per + 2 * grid, "flops": 0}
    if path in ("decimate", "preview"):
        return {"bytes": (n * 16 if path == "preview" else 16 * n // case["modulus"]) + 16 * n // case["modulus"],
                "flops": 0}
    if path == "spatial":
        return {"bytes": n * 16 + 16 * min(n, 1 << (3 * case["level"])) // 8, "flops": 0}
    if path == "digest":
        return {"bytes": n * 16, "flops": 0}
    if path == "render":
        return {"bytes": n * 16 // 4 + case["width"] * case["height"] * 8, "flops": 0}
    return {"bytes": n * (16 + 1 + 20), "flops": 0}


# ------------------------------------------------------------------ in 64 bits
def _mix(i):
    """splitmix64's first output for every seed in i (int64, wrapping)."""
    def shr(v, k):
        return (v >> k) & ((1 << (64 - k)) - 1)
    z = i - 0x61C8864680B583EB            # + 0x9E3779B97F4A7C15
    z = (z ^ shr(z, 30)) * -0x40A7B892E31B1A47   # 0xBF58476D1CE4E5B9
    z = (z ^ shr(z, 27)) * -0x6B2FB644ECCEEE15   # 0x94D049BB133111EB
    return z ^ shr(z, 31)


def _keeps(first, n, modulus):
    out = []
    for at in range(0, n, BLOCK):
        h = _mix(torch.arange(first + at, first + min(n, at + BLOCK), device="cuda", dtype=torch.int64))
        low = h & 0xFFFFFFFF
        high = (h >> 32) & 0xFFFFFFFF
        out.append(((high % modulus) * ((1 << 32) % modulus) + low) % modulus == 0)   # h mod m, h unsigned
    return torch.cat(out)


def _kept_count(n, first, modulus):
    return int(_keeps(first, n, modulus).sum())


def _cube(pts):
    lo, hi = pts[:, :3].amin(0).long(), pts[:, :3].amax(0).long()
    side = int((hi - lo).amax()) + 1
    return torch.cat([lo, hi, torch.tensor([side & 0xFFFFFFFF, side >> 32], device="cuda")]).to(torch.int32), lo, side


def exact(case, seed):
    """The previews in 64-bit torch; the octrees are whole numbers, compared as they are."""
    path = case["path"]
    if path not in ("decimate", "preview"):
        return None
    pts = cloud(case["cloud"], case["n"], seed)
    kept = pts[_keeps(case.get("first", 0), case["n"], case["modulus"])]
    out = torch.zeros((fp._preview_cap(case["n"], case["modulus"]), 4), dtype=torch.int32, device="cuda")
    out[:len(kept)] = kept
    count = torch.tensor([len(kept)], dtype=torch.int64, device="cuda")
    return [out, count] if path == "decimate" else [_cube(pts)[0], out, count]
