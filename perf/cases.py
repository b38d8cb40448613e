"""The work the library's speed is measured on: whole calls of its public
entry points over the sizes that its configurations, tests and benchmark use.

Every case is one call of a user's program on clouds that are already on the
GPU, with the context that such a program keeps.  The clouds are drawn on the
GPU from the seed alone, shaped like the repository's scenes: points uniform in
the KITTI detection range, spinning-LiDAR returns in scan order, and the
shuffled surface points of a furnished room.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2305_14306_gb300 import hav


def listed():
    return [
        # the smallest call: one object- or region-sized cloud, where launches and latency are all
        {"name": "tiny-1k", "kind": "chain", "scene": "room", "n": 1000, "levels": "250", "search": "bisect"},
        # the input stage of a point-based detector: one 16,384-point cloud, one level
        {"name": "uniform-16k", "kind": "chain", "scene": "box", "n": 16384, "levels": "4096", "search": "bisect"},
        # the set-abstraction stages of a LiDAR detector on one front view, as one chain
        {"name": "lidar-chain", "kind": "chain", "scene": "lidar", "n": 20876, "levels": "16384,4096,1024,512",
         "search": "bisect"},
        # indoor segmentation: a whole room, four levels of a quarter each
        {"name": "room-chain-1m", "kind": "chain", "scene": "room", "n": 1048576, "levels": "262144,65536,16384,4096",
         "search": "bisect"},
        # the same on a smaller room with the guided search start, ragged sizes
        {"name": "room-guided-300k", "kind": "chain", "scene": "room", "n": 300007, "levels": "75001,18750,4687",
         "search": "guided"},
        # a training batch of large LiDAR clouds of uneven size, two levels each
        {"name": "lidar-batch-64", "kind": "batch", "scene": "lidar", "clouds": 64, "lo": 20000, "hi": 200000,
         "levels": 2, "search": "bisect"},
        # a training batch of object-sized clouds, two levels each
        {"name": "small-batch-64", "kind": "batch", "scene": "box", "clouds": 64, "lo": 1000, "hi": 4000, "levels": 2,
         "search": "bisect"},
        # what a serving slot runs: requests of very different sizes and budgets packed into one call
        {"name": "served-mix-10", "kind": "batch", "scene": "served", "clouds": 10, "lo": 10000, "hi": 1000000,
         "levels": 1, "search": "bisect"},
        # grouping around sampled centres, the step that follows sampling in a set-abstraction block
        {"name": "group-room-64k", "kind": "group", "scene": "room", "n": 1048576, "m": 65536, "radius": 0.2,
         "nsample": 32},
        # farthest point sampling of a detector's input, the sampler this library is compared with
        {"name": "fps-16k", "kind": "fps", "scene": "box", "n": 16384, "m": 4096},
        # the spacing of a sampled subset with its histogram, the quality measure of a sampler
        {"name": "spacing-room-256k", "kind": "spacing", "scene": "room", "n": 1048576, "m": 262144, "bins": 24},
        # voxel means as representatives: one layer, coordinates beside the indices
        {"name": "xyz-mean-200k", "kind": "xyz", "scene": "lidar", "n": 200000, "m": 50000, "select": "mean"},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["chain", "chain", "chain", "batch", "batch", "batch", "group", "fps", "spacing", "xyz"])
    scene = rng.choice(["box", "lidar", "room"])
    search = rng.choice(["bisect", "bisect", "guided"])
    if kind == "chain":
        n = _log_int(rng, 700, 200000 if scene == "lidar" else 1048576)
        m, levels = n, []
        for _ in range(rng.randint(1, 4)):
            m = int(m * rng.uniform(0.2, 0.6))
            if m < 64:
                break
            levels.append(str(m))
        return {"kind": kind, "scene": scene, "n": n, "levels": ",".join(levels or [str(n // 4)]), "search": search}
    if kind == "batch":
        form = rng.randint(0, 2)
        if form == 0:
            return {"kind": kind, "scene": scene, "clouds": rng.randint(8, 96), "lo": 1000, "hi": 4000,
                    "levels": rng.randint(1, 2), "search": search}
        if form == 1:
            return {"kind": kind, "scene": "lidar", "clouds": rng.randint(4, 60), "lo": 20000,
                    "hi": _log_int(rng, 40000, 200000), "levels": rng.randint(1, 2), "search": search}
        return {"kind": kind, "scene": "served", "clouds": rng.randint(2, 12), "lo": 10000,
                "hi": _log_int(rng, 100000, 1000000), "levels": 1, "search": search}
    if kind == "group":
        n = _log_int(rng, 8000, 200000 if scene == "lidar" else 1048576)
        # radii that hold tens of points at the cloud's density
        scale = {"box": 2.0 * (16384 / n) ** (1 / 3), "lidar": 0.6 * math.sqrt(20000 / n),
                 "room": 0.1 * math.sqrt(1048576 / n)}[scene]
        return {"kind": kind, "scene": scene, "n": n, "m": max(64, n // rng.choice([4, 16, 64])),
                "radius": round(scale * rng.uniform(0.7, 2.0), 3), "nsample": rng.choice([16, 32, 64])}
    if kind == "fps":
        n = _log_int(rng, 1000, 100000)
        return {"kind": kind, "scene": scene, "n": n, "m": min(n // 2, rng.randint(256, 3500 if n <= 32768 else 1500))}
    if kind == "spacing":
        n = _log_int(rng, 4000, 200000 if scene == "lidar" else 1048576)
        return {"kind": kind, "scene": scene, "n": n, "m": max(1000, n // rng.choice([2, 4, 8])),
                "bins": rng.randint(8, 64)}
    n = _log_int(rng, 2000, 200000 if scene == "lidar" else 1048576)
    return {"kind": "xyz", "scene": scene, "n": n, "m": int(n * rng.uniform(0.05, 0.4)),
            "select": rng.choice(["mean", "centre"])}


# ------------------------------------------------------------------ clouds
def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _rand(g, *shape):
    return torch.rand(*shape, generator=g, device="cuda", dtype=torch.float64)


def _box_cloud(n, seed):
    """Uniform points in the KITTI detection range."""
    lo = torch.tensor([0.0, -40.0, -3.0], device="cuda", dtype=torch.float64)
    hi = torch.tensor([70.4, 40.0, 1.0], device="cuda", dtype=torch.float64)
    return (lo + (hi - lo) * _rand(_gen(seed), n, 3)).float().contiguous()


def _lidar_cloud(n, seed):
    """n returns, in scan order, of rings of rays over the front 90 degrees cast
    against the ground and 20 to 40 boxes, with 1 cm of range noise."""
    rng = np.random.default_rng(seed)
    g = _gen(seed)
    nb = int(rng.integers(20, 41))
    sides = rng.uniform(0.5, 4.0, (nb, 3))
    rad, ang = rng.uniform(5.0, 60.0, nb), np.deg2rad(rng.uniform(-45.0, 45.0, nb))
    c = np.stack([rad * np.cos(ang), rad * np.sin(ang)], axis=1)
    ground = -1.73
    lo = np.concatenate([c - sides[:, :2] / 2, np.full((nb, 1), ground)], axis=1)
    hi = np.concatenate([c + sides[:, :2] / 2, ground + sides[:, 2:]], axis=1)
    lo, hi = torch.from_numpy(lo).cuda(), torch.from_numpy(hi).cuda()
    rings = 64
    while True:
        steps = 2048 if n > 40000 else 512
        e = torch.deg2rad(torch.linspace(-24.9, 2.0, rings, device="cuda", dtype=torch.float64))
        a = torch.deg2rad(-45.0 + (torch.arange(steps, device="cuda", dtype=torch.float64) + 0.5) * 90.0 / steps)
        E, A = e.repeat_interleave(steps), a.repeat(rings)
        d = torch.stack([E.cos() * A.cos(), E.cos() * A.sin(), E.sin()], dim=1)
        t = torch.where(d[:, 2] < 0, ground / d[:, 2], math.inf)
        for b in range(nb):
            t1, t2 = lo[b] / d, hi[b] / d
            near, far = torch.minimum(t1, t2).amax(dim=1), torch.maximum(t1, t2).amin(dim=1)
            t = torch.where((near > 0) & (near <= far) & (near < t), near, t)
        t = t + 0.01 * torch.randn(t.shape, generator=g, device="cuda", dtype=torch.float64)
        ok = ((t > 0) & (t <= 80.0)).nonzero()[:, 0]
        if ok.numel() >= n:
            break
        rings *= 2
    ok = ok[torch.randperm(ok.numel(), generator=g, device="cuda")[:n]].sort().values
    return (d[ok] * t[ok, None]).float().contiguous()


def _room_cloud(n, seed):
    """Area-uniform points, shuffled, on the surfaces of a 10 x 10 x 3 m room
    with 30 to 60 boxes and panels, with 0.5 cm of noise."""
    rng = np.random.default_rng(seed)
    X, Y, Z = 10.0, 10.0, 3.0
    rects = [((0, 0, 0), (X, 0, 0), (0, Y, 0)), ((0, 0, Z), (X, 0, 0), (0, Y, 0)),
             ((0, 0, 0), (X, 0, 0), (0, 0, Z)), ((0, Y, 0), (X, 0, 0), (0, 0, Z)),
             ((0, 0, 0), (0, Y, 0), (0, 0, Z)), ((X, 0, 0), (0, Y, 0), (0, 0, Z))]
    for k in range(int(rng.integers(30, 61))):
        if k % 2 == 0:
            sx, sy, sz = rng.uniform(0.2, 2.0, 3)
            x, y = rng.uniform(0, X - sx), rng.uniform(0, Y - sy)
            rects += [((x, y, sz), (sx, 0, 0), (0, sy, 0)), ((x, y, 0), (sx, 0, 0), (0, 0, sz)),
                      ((x, y + sy, 0), (sx, 0, 0), (0, 0, sz)), ((x, y, 0), (0, sy, 0), (0, 0, sz)),
                      ((x + sx, y, 0), (0, sy, 0), (0, 0, sz))]
        else:
            a, b = rng.uniform(0.5, 3.0, 2)
            x, y, z = rng.uniform(0, X - a), rng.uniform(0, Y - b), rng.uniform(0, Z)
            h = min(a, Z - z)
            rects.append([((x, y, z), (a, 0, 0), (0, b, 0)), ((x, y, z), (0, b, 0), (0, 0, h)),
                          ((x, y, z), (a, 0, 0), (0, 0, h))][int(rng.integers(0, 3))])
    O, U, V = (torch.tensor([r[i] for r in rects], dtype=torch.float64, device="cuda") for i in range(3))
    cdf = torch.linalg.norm(torch.linalg.cross(U, V), dim=1).cumsum(0)
    g = _gen(seed)
    which = torch.searchsorted(cdf / cdf[-1], _rand(g, n), right=True).clamp_(max=len(rects) - 1)
    uv = _rand(g, n, 2)
    p = O[which] + uv[:, :1] * U[which] + uv[:, 1:] * V[which]
    p = p + 0.005 * torch.randn(p.shape, generator=g, device="cuda", dtype=torch.float64)
    return p.float().contiguous()


def _cloud(scene, n, seed):
    if scene == "served":  # scans up to 200,000 points, rooms above
        scene = "lidar" if n <= 200_000 else "room"
    return {"box": _box_cloud, "lidar": _lidar_cloud, "room": _room_cloud}[scene](n, seed)


def _batch_sizes(case):
    """Sizes spread over the case's range, in a mixed order, and the budgets of
    its levels (a quarter each; for served requests also a sixteenth or 4,096)."""
    S, lo, hi = case["clouds"], case["lo"], case["hi"]
    q = [((s * 0.6180339887498949) % 1.0) for s in range(1, S + 1)]
    n = [int(lo * (hi / lo) ** x) for x in q]
    if case["scene"] == "served":
        return n, [[(k // 4, k // 16, min(4096, k))[s % 3] for s, k in enumerate(n)]]
    m = [[k // 4 ** (j + 1) for k in n] for j in range(case["levels"])]
    return n, m


# ---------------------------------------------------------------- one call
def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        n, m = _batch_sizes(case)
        pts = torch.cat([_cloud(case["scene"], k, seed * 1000 + s) for s, k in enumerate(n)])
        return {"kind": kind, "ctx": hav.Context(sum(n), len(n)), "points": pts,
                "offsets": np.concatenate([[0], np.cumsum(n)]).astype(np.int64), "m": np.array(m, dtype=np.int64),
                "params": hav.params(search=case["search"])}
    pts = _cloud(case["scene"], case["n"], seed)
    st = {"kind": kind, "ctx": hav.Context(case["n"], 1), "points": pts}
    if kind == "chain":
        st["levels"] = [int(x) for x in case["levels"].split(",")]
        st["params"] = hav.params(search=case["search"])
    elif kind == "xyz":
        st["m"] = case["m"]
        st["params"] = hav.params(layers=1, select=case["select"])
    elif kind == "fps":
        st["m"] = case["m"]
    else:  # a subset of the points, ascending as the samplers return it
        idx = torch.randperm(case["n"], generator=_gen(seed + 77), device="cuda")[:case["m"]]
        st["idx"] = idx.sort().values.int()
        if kind == "group":
            st["radius"], st["nsample"] = case["radius"], case["nsample"]
        else:
            st["edges"] = _edges(case)
    return st


def _edges(case):
    """Ascending squared distances around the subset's mean spacing."""
    mean = {"box": (70.4 * 80.0 * 4.0 / case["m"]) ** (1 / 3), "lidar": 0.2, "room": math.sqrt(400.0 / case["m"])}
    return ((np.linspace(0.0, 3.0, case["bins"] + 1) * mean[case["scene"]]) ** 2).astype(np.float32)


def run(state):
    ctx, pts, kind = state["ctx"], state["points"], state["kind"]
    if kind == "chain":
        return hav.hav_sample_levels(ctx, pts, state["levels"], state["params"])
    if kind == "batch":
        return hav.hav_sample_batched(ctx, pts, state["offsets"], state["m"], state["params"])
    if kind == "group":
        return hav.hav_ball_query(ctx, pts, state["idx"], state["radius"], state["nsample"])
    if kind == "fps":
        return hav.hav_fps(ctx, pts, state["m"])
    if kind == "spacing":
        return hav.hav_spacing_histogram(ctx, pts, state["idx"], state["edges"])
    return hav.hav_sample_xyz(ctx, pts, state["m"], state["params"])


def work(case):
    kind = case["kind"]
    if kind == "batch":
        n, m = _batch_sizes(case)
        return {"bytes": 12 * sum(n) + 4 * sum(map(sum, m)), "flops": 12 * sum(n)}
    n = case["n"]
    if kind == "chain":
        m = [int(x) for x in case["levels"].split(",")]
        return {"bytes": 12 * n + 4 * sum(m), "flops": 12 * (n + sum(m[:-1]))}
    m = case["m"]
    if kind == "group":
        slots = m * case["nsample"]
        return {"bytes": 12 * n + 4 * m + 16 * slots, "flops": 8 * slots}
    if kind == "fps":
        return {"bytes": 12 * n + 4 * m, "flops": 8 * n}
    if kind == "spacing":
        return {"bytes": 12 * m + 4 * m + 4 * m + 8 * (case["bins"] + 2), "flops": 8 * m}
    return {"bytes": 12 * n + 16 * m, "flops": 12 * n}


# ------------------------------------------------- the same in 64 bits
def exact(case, seed):
    """Indices and counts have no 64-bit value; offsets, spacings and voxel
    means do.  Which points a ball, a voxel or a search step holds follows the
    library's definition in binary32 (single correctly rounded operations)."""
    kind = case["kind"]
    if kind == "group":
        st = prepare(case, seed)
        return None, _exact_group(st["points"], st["idx"].long(), st["radius"], st["nsample"])
    if kind == "spacing":
        st = prepare(case, seed)
        return _exact_spacing(st["points"][st["idx"].long()].double()), None
    if kind == "xyz":
        p = _cloud(case["scene"], case["n"], seed).cpu().numpy()
        return None, torch.from_numpy(_exact_representatives(p, case["m"], case["select"]))
    return None


def _exact_group(p, centres, radius, nsample):
    p64, r32 = p.double(), torch.tensor(radius, dtype=torch.float32, device="cuda")
    r2 = r32 * r32
    out = torch.empty(centres.numel(), nsample, 3, dtype=torch.float64, device="cuda")
    step = max(1, (1 << 27) // p.shape[0])
    for a in range(0, centres.numel(), step):
        c = p[centres[a:a + step]]
        d2 = torch.zeros(c.shape[0], p.shape[0], device="cuda")
        for k in range(3):
            e = p[None, :, k] - c[:, None, k]
            d2 += e * e
        row, col = (d2 < r2).nonzero(as_tuple=True)  # ascending indices within each row
        count = torch.bincount(row, minlength=c.shape[0])
        first = count.cumsum(0) - count
        slot = torch.arange(nsample, device="cuda")[None, :]
        take = first[:, None] + torch.where(slot < count[:, None], slot, 0)
        out[a:a + step] = p64[col[take]] - p64[centres[a:a + step]][:, None, :]
    return out.cpu()


def _exact_spacing(q):
    out = torch.empty(q.shape[0], dtype=torch.float64, device="cuda")
    step = max(1, (1 << 26) // q.shape[0])
    for a in range(0, q.shape[0], step):
        d2 = torch.zeros(min(step, q.shape[0] - a), q.shape[0], dtype=torch.float64, device="cuda")
        for k in range(3):
            d2 += (q[None, :, k] - q[a:a + step, None, k]) ** 2
        r = torch.arange(d2.shape[0], device="cuda")
        d2[r, a + r] = math.inf
        out[a:a + step] = d2.amin(dim=1)
    return out.cpu()


def _cells(p, s):
    f = np.floor(p / s)
    u = (f - np.floor(p.min(axis=0) / s)).astype(np.uint64)
    return f, u[:, 0] | u[:, 1] << np.uint64(21) | u[:, 2] << np.uint64(42)


def _exact_representatives(p, m, select):
    """One layer: bisection of the voxel size until m .. 1.05 m voxels are
    occupied, the m voxels of smallest SplitMix64 priority (or, with too few,
    the lowest other indices as themselves), and per index its voxel's centre
    or mean."""
    f32 = np.float32
    lo, hi = f32(0), (p.max(axis=0) - p.min(axis=0)).max()
    s = None
    for _ in range(20):
        mid = f32(f32(lo + hi) * f32(0.5))
        K = np.unique(_cells(p, mid)[1]).size
        if K > m + m * 5 // 100:
            lo = mid
        elif K < m:
            hi = mid
        else:
            s = mid
            break
    if s is None:
        s = lo if lo > 0 else hi
    f, key = _cells(p, s)
    d = p - s * (f + f32(0.5))
    d2 = (d[:, 0] * d[:, 0] + d[:, 1] * d[:, 1]) + d[:, 2] * d[:, 2]
    order = np.lexsort((np.arange(p.shape[0]), d2, key))
    uniq, first, inv, count = np.unique(key[order], return_index=True, return_inverse=True, return_counts=True)
    rep, p64 = order[first], p.astype(np.float64)
    mean = np.stack([np.bincount(inv, weights=p64[order, k], minlength=uniq.size) for k in range(3)], 1) / count[:, None]
    value = mean if select == "mean" else np.float64(s) * (f[rep].astype(np.float64) + 0.5)
    with np.errstate(over="ignore"):
        z = (uniq ^ (uniq >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
        z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
        z ^= z >> np.uint64(31)
    keep = np.argsort(z)[:m]
    out, taken = p64.copy(), np.zeros(p.shape[0], bool)
    out[rep[keep]] = value[keep]
    taken[rep[keep]] = True
    taken[np.nonzero(~taken)[0][:m - keep.size]] = True
    return out[taken]
