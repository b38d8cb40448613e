"""One cloud near the clusters' largest level: which kernel takes it depends on
the budget, the result does not; the following levels go to the clusters."""
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


# (points, budget, layers, extra parameters, launches of the call, and of one with clusters asked for or few blocks)
@pytest.mark.parametrize("n,m,layers,kw,launches", [
    (30000, [29000, 2100], 1, {}, (1, 1)),
    (30001, [11250, 2100], 1, {}, (1, 1)),
    (30001, [11251, 2100], 1, {}, (2, 1)),
    (32768, [28671, 2100], 2, {}, (1, 1)),
    (32768, [28672, 2100], 2, {}, (2, 1)),
    (32768, [32768, 3000], 2, {"search": "guided"}, (2, 1)),
    (32768, [32000], 1, {"select": "random", "seed": 4}, (1, 1)),
    (32768, [32000], 1, {"fixed_s": 0.05}, (1, 1)),
])
def test_budgets(hv, n, m, layers, kw, launches):
    pts = np.ascontiguousarray(scenes.room_scene(n, seed=n), dtype=np.float32)
    kw = dict(kw, layers=layers)
    (res, tro), = G.oracle_many([pts], [m], kw)
    p = hv.params(**kw)
    dev = torch.from_numpy(pts).cuda()
    ctx = hv.Context(n, 1)
    try:
        for ctas, blocks, count in ((0, 0, launches[0]), (0, 76, launches[0]), (0, 75, launches[1]), (16, 0, launches[1])):
            ctx.set_tuning(cluster_ctas=ctas, nblocks=blocks)
            before = ctx.launches()
            outs = hv.hav_sample_levels(ctx, dev, m, p)
            assert hv.hav_status_get(ctx, 1)[0] == 0
            assert ctx.launches() - before == count
            tr = hv.hav_trace_get(ctx, len(m) * layers)
            for j in range(len(m)):
                assert np.array_equal(outs[j].cpu().numpy(), res[j]), (ctas, j)
                for l in range(layers):
                    why = G.traces_equal(tr[j * layers + l], tro[j][l])
                    assert why is None, (ctas, j, l, why)
    finally:
        ctx.close()
