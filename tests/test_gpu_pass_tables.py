"""Several sizes a pass, so far apart that the coarse ones are counted with a
bit per cell and the fine ones with keys in one work item and not in another
(a few outliers among the first points of a dense cloud): the forms of a
size's table do not mix.  Indices and counts as the oracle's."""
import os
import sys

import numpy as np
import pytest

torch = pytest.importorskip("torch")
sys.path.insert(0, os.path.dirname(__file__))
import _gpu_helpers as G  # noqa: E402

pytestmark = pytest.mark.gpu

NEVER, ALWAYS = 0, 1 << 31
DEPTHS = {"three sizes": [NEVER, NEVER, ALWAYS], "seven sizes": [NEVER, ALWAYS, ALWAYS],
          "fifteen sizes": [ALWAYS, ALWAYS, ALWAYS]}


@pytest.fixture(scope="module")
def hv():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2305_14306_gb300 import build, hav
    build.build()
    hav.load()
    return hav


@pytest.mark.parametrize("table_log2", [1, 3])
@pytest.mark.parametrize("depth", DEPTHS)
@pytest.mark.parametrize("search", ["bisect", "guided"])
@pytest.mark.parametrize("n,wide", [(8193, 10), (20000, 10), (20000, 40), (32768, 10), (50000, 14)])
def test_outliers_in_one_item(hv, n, wide, search, depth, table_log2):
    rng = np.random.default_rng(n + wide)
    pts = rng.uniform(0, 100, (n, 3))
    first = rng.integers(0, 100, 25)
    pts[first] = rng.uniform(0, 100 * wide, (25, 3))
    pts = np.ascontiguousarray(pts, dtype=np.float32)
    kw = dict(search=search, layers=1)
    p = hv.params(**kw)
    dev = torch.from_numpy(pts).cuda()
    ctx = hv.Context(1 << 18, 1)
    try:
        ctx.set_tuning(small_points=0, solo_points=0, spec_points=DEPTHS[depth], table_log2=table_log2)
        for m in (n // 7, n // 25):
            (res, tro), = G.oracle_many([pts], [[m]], kw)
            for _ in range(2):  # (the second call starts on the tables the first one left)
                out = hv.hav_sample_levels(ctx, dev, [m], p)[0].cpu().numpy()
                assert hv.hav_status_get(ctx, 1)[0] == 0
                why = G.traces_equal(hv.hav_trace_get(ctx, 1)[0], tro[0][0])
                assert why is None, (m, why)
                assert np.array_equal(out, res[0]), m
    finally:
        ctx.close()


# a box of 2^21 cells and more along one axis and few along the others (keys, never
# bits): the call and an ordinary one after it on the same tables
@pytest.mark.parametrize("depth", [[NEVER, NEVER, NEVER], *DEPTHS.values()])
@pytest.mark.parametrize("search", ["bisect", "guided"])
@pytest.mark.parametrize("axis", [0, 1, 2])
def test_long_axis(hv, axis, search, depth):
    import oracle
    rng = np.random.default_rng(axis)
    long = rng.uniform(0, 1, (20000, 3)) * np.array([4e-3, 4e-3, 3e-3])
    long = long[rng.integers(0, 9000, 20000)]  # (repeats: never as many voxels as points)
    long[:, axis] = rng.uniform(0, 1e-3, 20000)[rng.integers(0, 9000, 20000)]
    long[77, axis], long[15000, axis] = 3000.0, 900.0
    box = rng.uniform(-5, 5, (30000, 3))
    clouds = [(np.ascontiguousarray(c, dtype=np.float32), m) for c, m in ((long, [19000]), (box, [20000, 4000]))]
    kw = dict(search=search)
    p = hv.params(**kw)
    ctx = hv.Context(1 << 17, 1)
    try:
        ctx.set_tuning(small_points=0, solo_points=0, spec_points=depth)
        for pts, m in (clouds[1], clouds[0], clouds[1], clouds[0], clouds[1]):
            outs = hv.hav_sample_levels(ctx, torch.from_numpy(pts).cuda(), m, p)
            status = hv.hav_status_get(ctx, 1)[0]
            try:
                (res, tro), = G.oracle_many([pts], [m], kw)
            except oracle.OracleError as e:
                assert status == e.status
                continue
            assert status == 0
            tr = hv.hav_trace_get(ctx, len(m) * p.layers)
            for j in range(len(m)):
                for l in range(p.layers):
                    why = G.traces_equal(tr[j * p.layers + l], tro[j][l])
                    assert why is None, (j, l, why)
                assert np.array_equal(outs[j].cpu().numpy(), res[j]), j
    finally:
        ctx.close()
