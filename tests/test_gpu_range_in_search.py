"""A voxel size that stops being representable in the middle of a search: the
cloud reports HAV_ERR_RANGE and gets its first indices, the other clouds of
the call are exact, and the context goes on, on every engine."""
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


def out_of_range(n, seed):
    """A few points, repeated, 1e16 from the origin: too few voxels at every
    size, and cell indices beyond 2^62 after some nine halvings."""
    rng = np.random.default_rng(seed)
    few = np.concatenate([np.full((5, 1), 1e16), rng.uniform(0, 1, (5, 2))], axis=1)
    return few[rng.integers(0, 5, n)]


@pytest.mark.parametrize("engine", ENGINES)
@pytest.mark.parametrize("search", ["bisect", "guided"])
@pytest.mark.parametrize("n", [60, 1000, 4000])
def test_range_in_the_search(hv, engine, search, n):
    import oracle
    kw = dict(search=search)
    bad = np.ascontiguousarray(out_of_range(n, n), dtype=np.float32)
    with pytest.raises(oracle.OracleError) as e:
        oracle.sample_levels(bad, [n // 2, n // 4], oracle.params(**kw))
    assert e.value.status == hv.HAV_ERR_RANGE
    healthy = [np.ascontiguousarray(scenes.room_scene(k, seed=k), dtype=np.float32) for k in (900, 2300, 3500)]
    p = hv.params(**kw)
    ctx = hv.Context(1 << 18, 256)
    try:
        ctx.set_tuning(**ENGINES[engine])
        for clouds in ([bad], [healthy[0], bad, healthy[1], bad, healthy[2]],
                       ([bad] * 3 + healthy) * (30 if n == 60 else 2)):
            levels = [[len(c) // 2, len(c) // 4] for c in clouds]
            want = dict(zip([900, 2300, 3500], G.oracle_many(healthy, [[k // 2, k // 4] for k in (900, 2300, 3500)], kw)))
            pts, offs = scenes.concat(clouds)
            m = np.array(levels, dtype=np.int64).T
            for _ in range(3):
                outs = [o.cpu().numpy() for o in hv.hav_sample_batched(ctx, torch.from_numpy(pts).cuda(), offs, m, p)]
                st, per = hv.hav_status_get(ctx, len(clouds))
                assert st == hv.HAV_ERR_RANGE
                for s, c in enumerate(clouds):
                    assert per[s] == (hv.HAV_ERR_RANGE if len(c) == n else 0), s
                    for j in range(2):
                        a = int(m[j, :s].sum())
                        res = np.arange(m[j, s]) if len(c) == n else want[len(c)][0][j]
                        assert np.array_equal(outs[j][a:a + m[j, s]], res), (s, j)
    finally:
        ctx.close()
