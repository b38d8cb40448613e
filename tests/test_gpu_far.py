"""Clouds whose voxels lie 2^20 to 2^24 cells from the origin (projected
coordinates with voxels a few steps of binary32 wide), on every engine:
indices and traces bit-identical to the oracle's."""
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
           "grid, one size": dict(small_points=0, solo_points=0, spec_points=[0, 0, 0]),
           "grid, three sizes": dict(small_points=0, solo_points=0, spec_points=[0, 0, 1 << 31])}


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


def check(hv, ctx, clouds, levels, engines=ENGINES, **pkw):
    clouds = [np.ascontiguousarray(c, dtype=np.float32) for c in clouds]
    want = G.oracle_many(clouds, levels, pkw)
    pts, offs = scenes.concat(clouds)
    dev = torch.from_numpy(pts).cuda()
    m = np.array(levels, dtype=np.int64).T
    p = hv.params(**pkw)
    for name in engines:
        if max(len(c) for c in clouds) > (4096 if name == "one CTA" else 1 << 18 if "grid" in name else 32768):
            continue
        ctx.set_tuning(**ENGINES[name])
        outs = [o.cpu().numpy() for o in hv.hav_sample_batched(ctx, dev, offs, m, p)]
        assert hv.hav_status_get(ctx, len(clouds))[0] == 0, name
        tr = hv.hav_trace_get(ctx, m.size * p.layers)
        for s, (res, tro) in enumerate(want):
            for j in range(m.shape[0]):
                a = int(m[j, :s].sum())
                assert np.array_equal(outs[j][a:a + m[j, s]], res[j]), (name, s, j)
                for l in range(p.layers):
                    why = G.traces_equal(tr[(j * len(clouds) + s) * p.layers + l], tro[j][l])
                    assert why is None, (name, s, j, l, why)


def far_cloud(n, m, voxels, seed):
    """A uniform box whose voxels at budget m lie about 2^voxels cells away, along x, y or both."""
    rng = np.random.default_rng(seed)
    side = m ** (1 / 3)  # cells of the box along an axis at that size, of width 1
    at = 2.0 ** abs(voxels) * rng.uniform(1, 1.3) * np.sign(voxels)
    return rng.uniform(0, side, (n, 3)) + np.array([[at, 0, 0], [0, -at, 0], [at, at, 5]][seed % 3])


@pytest.mark.parametrize("voxels", [20, -20, 20.7, 21, -21, 21.5, 21.9, -21.9, 22, -22, 22.3, 22.6, -23, 24])
@pytest.mark.parametrize("n", [3000, 20000, 60000])
def test_far(hv, ctx, voxels, n):
    seed = n + int(10 * abs(voxels))
    cloud = far_cloud(n, n // 4, voxels, seed)
    check(hv, ctx, [cloud], [[n // 4, n // 20]])
    check(hv, ctx, [cloud], [[n // 6]], search="guided", layers=1, select="random", seed=3)


def test_far_and_near_in_a_batch(hv, ctx):
    clouds = [far_cloud(3000, 700, 22.2, 1), scenes.uniform_box(2500, 2), far_cloud(4000, 900, -21.7, 3),
              scenes.room_scene(1200, 4)]
    check(hv, ctx, clouds, [[len(c) // 4, len(c) // 10] for c in clouds])


# boxes of up to 2^21 cells along an axis at the one size, from far to near
@pytest.mark.parametrize("lo,hi", [(-4194320, -2200000), (2200000, 4194330), (-1048570, 1048560), (1048000, 3000000)])
def test_long_boxes(hv, ctx, lo, hi):
    rng = np.random.default_rng(4)
    cloud = rng.uniform([lo, -5, 2], [hi, 5, 9], (4000, 3))
    check(hv, ctx, [cloud], [[1500]], layers=1, fixed_s=1.0)
    cloud = np.repeat(np.rint(cloud[:500]), 8, axis=0)
    check(hv, ctx, [cloud], [[300]], layers=1, fixed_s=1.0)
