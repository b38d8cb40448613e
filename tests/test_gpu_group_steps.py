"""The ball query's grid of cells and index steps, and the spacing search over
it, against the oracle at the edges of both."""
import contextlib
import os
import sys

import numpy as np
import pytest

torch = pytest.importorskip("torch")
sys.path.insert(0, os.path.dirname(__file__))
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


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a, dtype=np.float32)).cuda()


def check(hv, oracle_mod, pts, centres, radius, nsample, room=None):
    """room: points the context holds (its scratch bounds cells and steps)."""
    centres = np.ascontiguousarray(centres, dtype=np.int32)
    with contextlib.closing(hv.Context(room or len(pts), 1)) as ctx:
        idx, xyz = hv.hav_ball_query(ctx, dev(pts), torch.from_numpy(centres).cuda(), radius, nsample)
        assert hv.hav_status_get(ctx, 1)[0] == 0
    o_idx, o_xyz = oracle_mod.ball_query(pts, centres, radius, nsample)
    assert np.array_equal(idx.cpu().numpy(), o_idx)
    assert np.array_equal(xyz.cpu().numpy().view(np.uint32), o_xyz.view(np.uint32))


# fewer points than steps, one step's edge, and enough for several rounds of steps
@pytest.mark.parametrize("n", [1, 2, 15, 16, 17, 33, 255, 257, 4097, 30000])
@pytest.mark.parametrize("nsample", [1, 31, 128, 129, 256])
def test_sizes(hv, oracle_mod, n, nsample):
    pts = scenes.uniform_box(n, seed=n)
    side = float(np.ptp(pts, axis=0).max()) if n > 1 else 1.0
    check(hv, oracle_mod, pts, np.arange(0, n, max(1, n // 97)), max(side * 0.3, 1e-3), nsample)


@pytest.mark.parametrize("radius", [1e-4, 0.03, 0.6, 40.0])
@pytest.mark.parametrize("room", [None, 1 << 18])
def test_radii(hv, oracle_mod, radius, room):
    pts = scenes.room_scene(20000, seed=5)
    check(hv, oracle_mod, pts, np.arange(0, 20000, 83), radius, 24, room)


@pytest.mark.parametrize("form", ["same", "halves", "reversed", "late", "plane", "lattice", "not finite", "vast"])
def test_forms(hv, oracle_mod, form):
    rng = np.random.default_rng(6)
    box = scenes.uniform_box(6000, 7)
    lattice = np.stack(np.meshgrid(*[np.arange(17)] * 3, indexing="ij"), -1).reshape(-1, 3)
    centres = np.arange(0, 4000, 41)
    pts, radius = {
        "same": lambda: (np.ones((5000, 3)), 0.5),
        # every qualifying point in the first or the last index steps
        "halves": lambda: (np.concatenate([box[:4000], box[:4000] + 1e3]), 9.0),
        "reversed": lambda: (box[np.argsort(-box[:, 0])], 9.0),
        "late": lambda: (np.concatenate([box[:4000] * 50, np.repeat(box[:1] * 50, 3000, 0)]), 9.0),
        "plane": lambda: (box * [1, 1, 0], 4.0),
        "lattice": lambda: (lattice, 2.0),
        "not finite": lambda: (np.concatenate([box, np.where(rng.random((500, 3)) < 0.4, np.nan, box[:500]),
                                               np.full((40, 3), np.inf)]), 9.0),
        "vast": lambda: (np.concatenate([box, [[3e38, 0, 0], [-3e38, 0, 0]]]), 9.0),
    }[form]()
    pts = np.ascontiguousarray(pts, dtype=np.float32)
    for nsample in (3, 40, 256):
        check(hv, oracle_mod, pts, centres, radius, nsample)


@pytest.mark.parametrize("form", ["box", "line", "plane", "twice", "clusters", "not finite", "vast"])
def test_spacing(hv, oracle_mod, form):
    box = scenes.uniform_box(32768, 8)
    pts = {"box": lambda: box,
           "line": lambda: box * [1, 0, 0],
           "plane": lambda: box * [0, 1, 1],
           "twice": lambda: np.concatenate([box[:16384]] * 2),
           "clusters": lambda: np.concatenate([box[:20000] * 1e-3, box[:12768] * 1e-3 + 40]),
           "not finite": lambda: np.where(np.arange(32768)[:, None] % 9 == 0, [[0, np.inf, np.nan]], box),
           "vast": lambda: np.concatenate([box[:32766], [[3e38, 0, 0], [-3e38, 0, 0]]])}[form]()
    pts = np.ascontiguousarray(pts, dtype=np.float32)
    idx = np.random.default_rng(9).permutation(32768).astype(np.int32)
    with contextlib.closing(hv.Context(32768, 1)) as ctx:
        got = hv.hav_spacing(ctx, dev(pts), torch.from_numpy(idx).cuda())
        assert hv.hav_status_get(ctx, 1)[0] == 0
    assert np.array_equal(got.cpu().numpy().view(np.uint32), oracle_mod.spacing(pts, idx).view(np.uint32))


# one range of candidates and its neighbours, and the line between all pairs and the grid
@pytest.mark.parametrize("m", [1, 2, 31, 32, 33, 255, 1023, 1024, 1025, 9001, 24575, 24576, 24577])
def test_spacing_sizes(hv, oracle_mod, m):
    pts = scenes.room_scene(30000, seed=3)
    idx = np.random.default_rng(m).permutation(30000)[:m].astype(np.int32)
    with contextlib.closing(hv.Context(30000, 1)) as ctx:
        got = hv.hav_spacing(ctx, dev(pts), torch.from_numpy(idx).cuda())
        assert hv.hav_status_get(ctx, 1)[0] == 0
    assert np.array_equal(got.cpu().numpy().view(np.uint32), oracle_mod.spacing(pts, idx).view(np.uint32))
