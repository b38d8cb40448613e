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
