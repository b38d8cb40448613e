"""The grid kernel's bisection passes where their ways to count change: tiles
of an item, hashed and direct words, keys, bits per cell and the sort of a
batch's segments; indices and traces bit-identical to the oracle's."""
import os
import sys

import numpy as np
import pytest

torch = pytest.importorskip("torch")
sys.path.insert(0, os.path.dirname(__file__))
import _gpu_helpers as G  # noqa: E402
from paper_2305_14306_gb300 import scenes  # noqa: E402

pytestmark = pytest.mark.gpu

NEVER, ALWAYS = 0, 1 << 31
SHAPES = {"one size": dict(spec_points=[NEVER, NEVER, NEVER]),
          "three sizes": dict(spec_points=[NEVER, NEVER, ALWAYS]),
          "seven sizes, two probes": dict(spec_points=[NEVER, ALWAYS, ALWAYS], pass_shape=2),
          "several tiles an item": dict(spec_points=[NEVER, NEVER, NEVER], nblocks=3)}


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
    c = hv.Context(1 << 18, 8)
    yield c
    c.close()


def scattered(n, spread, seed):
    rng = np.random.default_rng(seed)
    return rng.normal(0, 1, (n, 3)) + rng.integers(0, 4, (n, 1)) * np.array([spread, -spread, spread / 3])


CLOUDS = {
    # the shortest sorted segment and its neighbours, an empty and a tiny one
    "sort edge": lambda: [scenes.room_scene(n, seed=n) for n in (16383, 16384, 16385)] + [
        np.zeros((0, 3)), scenes.uniform_box(5, 1)],
    # more points than eight tiles of three blocks hold
    "large": lambda: [scenes.room_scene(230_000, seed=3)],
    "scan": lambda: [scenes.lidar_exact(60_000, 4)],
    "lattice": lambda: [np.random.default_rng(5).integers(-40, 41, (50_000, 3)) * 0.125],
    "flat": lambda: [scenes.uniform_box(40_000, 6) * np.array([1, 1, 0])],
    # boxes of 2^30 cells and more at the sizes the search visits
    "far apart": lambda: [scattered(40_000, 4000.0, 7)],
    "farther apart": lambda: [scattered(40_000, 60000.0, 8), scenes.uniform_box(20_000, 9)],
    "offset": lambda: [scenes.uniform_box(33_000, 10) + np.array([-7000, 9000, 500])],
    "copies": lambda: [np.repeat(scenes.uniform_box(900, 11), 40, axis=0)],
}


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("cloud", CLOUDS)
def test_passes(hv, ctx, cloud, shape):
    import oracle
    clouds = [np.ascontiguousarray(c, dtype=np.float32) for c in CLOUDS[cloud]()]
    levels = [[len(c) // 4, len(c) // 9] for c in clouds]
    status = 0
    try:
        want = G.oracle_many(clouds, levels)
    except oracle.OracleError as e:
        want, status = [], e.status
    pts, offs = scenes.concat(clouds)
    ctx.set_tuning(nblocks=0)
    ctx.set_tuning(small_points=0, solo_points=0, pass_shape=0)
    ctx.set_tuning(**SHAPES[shape])
    p = hv.params()
    m = np.array(levels, dtype=np.int64).T
    for _ in range(2):  # (the second call starts on the tables the first one left)
        outs = [o.cpu().numpy() for o in hv.hav_sample_batched(ctx, torch.from_numpy(pts).cuda(), offs, m, p)]
        st, _ = hv.hav_status_get(ctx, len(clouds))
        assert st == status
        tr = hv.hav_trace_get(ctx, m.size * p.layers)
        for s, (res, tro) in enumerate(want):
            for j in range(2):
                a = int(m[j, :s].sum())
                assert np.array_equal(outs[j][a:a + m[j, s]], res[j]), (s, j)
                for l in range(p.layers):
                    why = G.traces_equal(tr[(j * len(clouds) + s) * p.layers + l], tro[j][l])
                    assert why is None, (s, j, l, why)


# a level one point short of the size from which its short segments are sorted, and at it
@pytest.mark.parametrize("total", [(1 << 19) - 1, 1 << 19])
def test_sort_line(hv, total):
    short = [scenes.room_scene(n, seed=n) for n in (16383, 16384, 16385)] + [scenes.uniform_box(5, 1)]
    clouds = short + [scenes.uniform_box(total - sum(len(c) for c in short), 2)]
    clouds = [np.ascontiguousarray(c, dtype=np.float32) for c in clouds]
    levels = [[len(c) // 4] for c in clouds]
    want = G.oracle_many(clouds, levels)
    pts, offs = scenes.concat(clouds)
    c = hv.Context(total, len(clouds))
    try:
        c.set_tuning(small_points=0, solo_points=0)
        m = np.array(levels, dtype=np.int64).T
        out = hv.hav_sample_batched(c, torch.from_numpy(pts).cuda(), offs, m, hv.params())[0].cpu().numpy()
        assert hv.hav_status_get(c, len(clouds))[0] == 0
    finally:
        c.close()
    for s, (res, _) in enumerate(want):
        a = int(m[0, :s].sum())
        assert np.array_equal(out[a:a + m[0, s]], res[0]), s


# candidates of the bin that the cut-off falls in: none, one, up to a warp's lanes and many more, in several segments
@pytest.mark.parametrize("sizes", [[900], [40_000], [150_000], [70_000, 300, 33_000]])
@pytest.mark.parametrize("part", [1, 2, 5, 97])
def test_cut_off(hv, ctx, sizes, part):
    clouds = [np.ascontiguousarray(scenes.uniform_box(n, seed=n), dtype=np.float32) for n in sizes]
    levels = [[max(1, len(c) * 6 // 10 // part)] for c in clouds]
    kw = dict(layers=1, fixed_s=0.3)  # nearly every point in a voxel of its own
    want = G.oracle_many(clouds, levels, kw)
    pts, offs = scenes.concat(clouds)
    ctx.set_tuning(nblocks=0)
    ctx.set_tuning(small_points=0, solo_points=0, pass_shape=0)
    m = np.array(levels, dtype=np.int64).T
    out = hv.hav_sample_batched(ctx, torch.from_numpy(pts).cuda(), offs, m, hv.params(**kw))[0].cpu().numpy()
    assert hv.hav_status_get(ctx, len(clouds))[0] == 0
    for s, (res, _) in enumerate(want):
        a = int(m[0, :s].sum())
        assert np.array_equal(out[a:a + m[0, s]], res[0]), s
