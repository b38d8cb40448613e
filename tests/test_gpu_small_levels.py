"""The small-level kernels (one CTA, 8- and 16-CTA clusters) at the sizes where
their splits change and on clouds that reach every way a pass counts: indices
and traces bit-identical to the oracle's."""
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
           "16 CTAs": dict(small_points=32768, solo_points=0, cluster_ctas=16)}


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
    c = hv.Context(1 << 16, 64)
    yield c
    c.close()


def check(hv, ctx, clouds, levels, **pkw):
    """Every engine that takes the clouds, alone and (several) as a batch.  A
    cloud whose cells leave the key range reports what the oracle reports."""
    import oracle
    pts, offs = scenes.concat(clouds)
    m = np.array(levels, dtype=np.int64).T  # [level][cloud]
    status = 0
    try:
        want = G.oracle_many(clouds, levels, pkw)
    except oracle.OracleError as e:
        want, status = [], e.status
    p = hv.params(**pkw)
    for name, tune in ENGINES.items():
        if name == "one CTA" and max(len(c) for c in clouds) > 4096:
            continue
        ctx.set_tuning(**tune)
        outs = [o.cpu().numpy() for o in hv.hav_sample_batched(
            ctx, torch.from_numpy(pts).cuda(), offs, m, p)]
        st, _ = hv.hav_status_get(ctx, len(clouds))
        assert st == status, (name, st)
        tr = hv.hav_trace_get(ctx, m.size * p.layers)
        for s, (res, tro) in enumerate(want):
            for j in range(m.shape[0]):
                a = int(m[j, :s].sum())
                assert np.array_equal(outs[j][a:a + m[j, s]], res[j]), (name, s, j)
                for l in range(p.layers):
                    why = G.traces_equal(tr[(j * len(clouds) + s) * p.layers + l], tro[j][l])
                    assert why is None, (name, s, j, l, why)


# a warp, a stride of the counting threads (480 on one CTA, 512), the copy in
# shared memory (4,096) and the largest level, each with its neighbours
@pytest.mark.parametrize("n", [1, 2, 31, 33, 479, 480, 481, 511, 513, 1025, 2049, 4095, 4096, 4097, 8193, 16385, 32767,
                               32768])
def test_sizes(hv, ctx, n):
    cloud = scenes.room_scene(n, seed=n)
    check(hv, ctx, [cloud], [[max(1, n // 3), max(1, n // 7)]])
    check(hv, ctx, [cloud], [[n]], layers=1)


def lattice(n, pitch, seed):
    """Points at multiples of pitch (exact quotients at the bisection's sizes), both signs, with repeats."""
    rng = np.random.default_rng(seed)
    return (rng.integers(-16, 17, size=(n, 3)) * pitch).astype(np.float32)


def scattered(n, spread, seed):
    """Clusters so far apart that the box spans far more cells than any table
    holds: 2^18 to 2^40 cells at the sizes the search visits."""
    rng = np.random.default_rng(seed)
    return (rng.normal(0, 1, (n, 3)) + rng.integers(0, 4, (n, 1)) * np.array([spread, -spread, spread / 3])).astype(
        np.float32)


@pytest.mark.parametrize("search", ["bisect", "guided"])
@pytest.mark.parametrize("cloud", ["lattice", "third", "axis", "scattered", "far scattered", "offset", "same"])
def test_forms(hv, ctx, cloud, search):
    n = 3000
    pts = {"lattice": lambda: lattice(n, 0.25, 1),
           "third": lambda: lattice(n, np.float32(1 / 3), 2),
           "axis": lambda: scenes.uniform_box(n, 3) * np.array([1, 0, 1], np.float32),  # a flat cloud at y = 0
           "scattered": lambda: scattered(n, 300.0, 4),
           "far scattered": lambda: scattered(n, 20000.0, 5),
           "offset": lambda: scenes.uniform_box(n, 6) + np.array([4000, -9000, 300], np.float32),
           "same": lambda: np.repeat(scenes.uniform_box(5, 7), n // 5, axis=0)}[cloud]()
    pts = np.ascontiguousarray(pts, dtype=np.float32)
    check(hv, ctx, [pts], [[700, 100]], search=search)
    check(hv, ctx, [pts], [[2000]], search=search, t_max=7, layers=1, select="random", seed=9)


def test_large_forms_and_batches(hv, ctx):
    check(hv, ctx, [scattered(20000, 5000.0, 8)], [[9000, 800]])
    check(hv, ctx, [lattice(30000, 0.5, 9)], [[5000, 64]])
    clouds = [scenes.uniform_box(k, 10 + k) for k in (1, 40, 700, 2500, 4096)] + [lattice(1500, 0.125, 3)]
    check(hv, ctx, clouds, [[max(1, len(c) // 4), max(1, len(c) // 16)] for c in clouds])


# most points in a voxel of their own, with few and with many cells per slot of a pass
@pytest.mark.parametrize("n,m", [(4096, 4000), (9000, 8900), (20000, 19500), (32768, 31000), (32768, 32700)])
def test_crowded_passes(hv, ctx, n, m):
    check(hv, ctx, [scenes.uniform_box(n, n)], [[m]], layers=1)
    check(hv, ctx, [scattered(n, 2000.0, m)], [[m]], layers=1)
