"""Searches at sizes where the box spans 2^32 cells and more (small-level
kernels): cells whose numbers agree modulo 2^32 or whose table entries look
alike, scans at nearly every point a voxel, outliers.  Indices and traces
bit-identical to the oracle's on every engine."""
import os
import sys

import numpy as np
import pytest

torch = pytest.importorskip("torch")
sys.path.insert(0, os.path.dirname(__file__))
import _gpu_helpers as G  # noqa: E402
from paper_2305_14306_gb300 import scenes  # noqa: E402

pytestmark = pytest.mark.gpu

ENGINES = {"one CTA": dict(small_points=0, solo_points=4096),
           "8 CTAs": dict(small_points=32768, solo_points=0, cluster_ctas=8),
           "16 CTAs": dict(small_points=32768, solo_points=0, cluster_ctas=16),
           "grid": dict(small_points=0, solo_points=0)}


@pytest.fixture(scope="module")
def hv():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2305_14306_gb300 import build, hav
    build.build()
    hav.load()
    return hav


@pytest.fixture(scope="module")
def ctx(hv):
    c = hv.Context(1 << 16, 8)
    yield c
    c.close()


def check(hv, ctx, pts, levels, **pkw):
    pts = np.ascontiguousarray(pts, dtype=np.float32)
    (res, tro), = G.oracle_many([pts], [levels], pkw)
    p = hv.params(**pkw)
    dev = torch.from_numpy(pts).cuda()
    for name, tune in ENGINES.items():
        if name == "one CTA" and len(pts) > 4096:
            continue
        ctx.set_tuning(**tune)
        outs = hv.hav_sample_levels(ctx, dev, levels, p)
        assert hv.hav_status_get(ctx, 1)[0] == 0, name
        tr = hv.hav_trace_get(ctx, len(levels) * p.layers)
        for j in range(len(levels)):
            assert np.array_equal(outs[j].cpu().numpy(), res[j]), (name, j)
            for l in range(p.layers):
                why = G.traces_equal(tr[j * p.layers + l], tro[j][l])
                assert why is None, (name, j, l, why)
    return tro


def unmix(h):
    """The keys whose hash (slot_mix) is h: its steps backwards."""
    inverse = np.uint64(pow(0xD6E8FEB86659FD93, -1, 1 << 64))
    h ^= h >> np.uint64(32)
    h = h * inverse
    h ^= h >> np.uint64(32)
    h = h * inverse
    return h ^ (h >> np.uint64(32))


def alike(want, seed):
    """Cells with indices below 2^16 whose entries have the same 16 bits and whose
    probes start within 1/256 of the table from one another."""
    rng = np.random.default_rng(seed)
    found = np.zeros((0, 3), dtype=np.int64)
    while len(found) < want:
        h = rng.integers(0, 1 << 40, 1 << 20, dtype=np.uint64)
        # bits 56..63: where the probes start; 32..47: the entry's 16 bits
        low = h & np.uint64(0xFFFFFFFF)
        key = unmix(np.uint64(0x5A) << np.uint64(56) | (h >> np.uint64(32)) << np.uint64(48) |
                    np.uint64(0xBEEF) << np.uint64(32) | low)
        cells = np.stack([(key >> np.uint64(21 * a)) & np.uint64(0x1FFFFF) for a in range(3)], 1).astype(np.int64)
        ok = (cells < 65530).all(1) & (cells > 4).all(1) & (key >> np.uint64(63) == 0)
        found = np.concatenate([found, cells[ok]])
    return found[:want]


# at size E / 2^16 of a cube of side E (step 16 of the search) the box has 65,537 cells an axis
@pytest.mark.parametrize("cells,others,repeats", [(40, 10, 1), (40, 300, 4), (300, 900, 3), (300, 9000, 2), (600, 25000, 5)])
def test_entries_alike(hv, ctx, cells, others, repeats):
    rng = np.random.default_rng(cells + others)
    side = float(2**16 - 1)
    s = side / 2**16
    at = np.concatenate([alike(cells, cells)] * repeats)
    pts = np.concatenate([[[0, 0, 0], [side, side, side]], (at + rng.uniform(0.3, 0.7, at.shape)) * s,
                          rng.uniform(0, side, (others, 3))])
    pts = np.concatenate([pts, pts[-5:]])[rng.permutation(len(pts) + 5)]
    tro = check(hv, ctx, pts, [len(pts)], layers=1)  # (never enough voxels: every size of the search)
    assert int(tro[0][0]["iters"]) == 20
    check(hv, ctx, pts, [cells + others], sigma=(0, 1))
    check(hv, ctx, pts, [(cells + others) // 2], search="guided")


def twins(pairs, repeats, seed):
    """A cube of side E = 2^16 - 1 with pairs of points (1, -2, 1) E / 2^16
    apart.  At size E / 2^t, t >= 16, the box has 2^t + 1 cells an axis and the
    two cells' numbers differ by ((2^t)^2) 2^(t - 16), a multiple of 2^32."""
    rng = np.random.default_rng(seed)
    side = float(2**16 - 1)
    s = side / 2**16
    a = rng.integers(8, 2**16 - 8, (pairs, 3)) * s + 0.5 * s
    b = a + np.array([1, -2, 1]) * s
    close = a[: pairs // 8] + np.array([0.2, 0, 0.1]) * s  # apart from some t = 18 on
    corners = np.array([[0, 0, 0], [side, side, side]], dtype=np.float64)
    # cells 2^32 - 1 at t = 16: (0, 65535, 0)
    marked = np.tile([[0.25 * s, 65535.5 * s, 0.25 * s]], (3, 1))
    pts = np.concatenate([corners, marked, close] + [a, b] * repeats)
    return pts[rng.permutation(len(pts))]


# cells whose numbers agree modulo 2^32: few, and more than are collected
@pytest.mark.parametrize("pairs,repeats", [(3, 3), (900, 2), (1900, 1), (200, 30), (900, 8), (5000, 2), (15000, 1)])
def test_twins(hv, ctx, pairs, repeats):
    pts = twins(pairs, repeats, pairs)
    tro = check(hv, ctx, pts, [len(pts)], layers=1)  # (never enough voxels: every size of the search)
    assert int(tro[0][0]["iters"]) == 20
    check(hv, ctx, pts, [2 * pairs + 3 + pairs // 16], sigma=(0, 1), layers=1)
    check(hv, ctx, pts, [pairs + pairs // 2, pairs // 3], search="guided")


@pytest.mark.parametrize("n,m", [(4096, 4000), (12000, 11900), (20000, 18000), (32768, 31000), (32768, 32700)])
def test_scans(hv, ctx, n, m):
    check(hv, ctx, scenes.lidar_exact(n, n), [m], layers=1)
    check(hv, ctx, scenes.lidar_exact(n, n + 1), [m, m // 2])


# a dense cloud and one point far away: many points a cell, 2^36 cells and more
@pytest.mark.parametrize("n", [3000, 20000, 32000])
def test_one_outlier(hv, ctx, n):
    pts = scenes.room_scene(n, seed=n)
    pts[n // 3] = [30000, -20000, 25000]
    check(hv, ctx, pts, [n // 4, n // 16])
    check(hv, ctx, pts, [n // 2], layers=1, search="guided")
