"""Passes of the grid kernel in which a work item both holds voxels whole and
has undecided units (hashed words): the two share a list.  Indices and counts
as the oracle's, call after call."""
import os
import sys

import numpy as np
import pytest

torch = pytest.importorskip("torch")
sys.path.insert(0, os.path.dirname(__file__))
import _gpu_helpers as G  # noqa: E402
from paper_2305_14306_gb300 import scenes  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def hv():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2305_14306_gb300 import build, hav
    build.build()
    hav.load()
    return hav


# sorted clouds whose items span more cells than words at the sizes near the end of the search
@pytest.mark.parametrize("depth", [[0, 0, 0], [0, 0, 1 << 31]])
@pytest.mark.parametrize("cloud,m", [("room", [140_000, 60_000]), ("box", [150_000, 100_000]), ("scan", [120_000])])
def test_owned_beside_undecided(hv, cloud, m, depth):
    n = 160_000
    pts = {"room": lambda: scenes.room_scene(n, seed=1), "box": lambda: scenes.uniform_box(n, 2),
           "scan": lambda: scenes.lidar_exact(n, 3)}[cloud]()
    pts = np.ascontiguousarray(pts, dtype=np.float32)
    (res, tro), = G.oracle_many([pts], [m])
    dev = torch.from_numpy(pts).cuda()
    p = hv.params()
    ctx = hv.Context(1 << 20, 1)
    try:
        ctx.set_tuning(small_points=0, solo_points=0, spec_points=depth)
        for _ in range(12):
            outs = hv.hav_sample_levels(ctx, dev, m, p)
            assert hv.hav_status_get(ctx, 1)[0] == 0
            tr = hv.hav_trace_get(ctx, len(m) * p.layers)
            for j in range(len(m)):
                assert np.array_equal(outs[j].cpu().numpy(), res[j]), j
                for l in range(p.layers):
                    why = G.traces_equal(tr[j * p.layers + l], tro[j][l])
                    assert why is None, (j, l, why)
    finally:
        ctx.close()


# extents so small that the sorting cells' scale 16 / extent overflows (or hardly does not): nothing is owned
@pytest.mark.parametrize("extent", [2e-38, 4.6e-38, 6e-38])
@pytest.mark.parametrize("sizes", [[140_000], [30_000, 60_000, 440_000]])
def test_sorted_tiny_extents(hv, sizes, extent):
    rng = np.random.default_rng(7)
    clouds = [np.ascontiguousarray(rng.uniform(0, extent, (n, 3)), dtype=np.float32) for n in sizes[:2]]
    clouds += [scenes.uniform_box(n, n) for n in sizes[2:]]
    levels = [[len(c) // 3, len(c) // 10] for c in clouds]
    want = G.oracle_many(clouds, levels)
    pts, offs = scenes.concat(clouds)
    m = np.array(levels, dtype=np.int64).T
    p = hv.params()
    ctx = hv.Context(int(offs[-1]), len(clouds))
    try:
        ctx.set_tuning(small_points=0, solo_points=0)
        outs = [o.cpu().numpy() for o in hv.hav_sample_batched(ctx, torch.from_numpy(pts).cuda(), offs, m, p)]
        assert hv.hav_status_get(ctx, len(clouds))[0] == 0
        tr = hv.hav_trace_get(ctx, m.size * p.layers)
    finally:
        ctx.close()
    for s, (res, tro) in enumerate(want):
        for j in range(2):
            for l in range(p.layers):
                why = G.traces_equal(tr[(j * len(clouds) + s) * p.layers + l], tro[j][l])
                assert why is None, (s, j, l, why)
            a = int(m[j, :s].sum())
            assert np.array_equal(outs[j][a:a + m[j, s]], res[j]), (s, j)
