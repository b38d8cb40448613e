"""Farthest point sampling on one cluster, many picks per barrier: the oracle's
sequence of picks on clouds where lists are short, long, tied or empty."""
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


@pytest.fixture(scope="module")
def ctx(hv):
    c = hv.Context(1 << 18, 1)
    yield c
    c.close()


def check(hv, ctx, oracle_mod, pts, m):
    pts = np.ascontiguousarray(pts, dtype=np.float32)
    got = hv.hav_fps(ctx, torch.from_numpy(pts).cuda(), m).cpu().numpy()
    st, _ = hv.hav_status_get(ctx, 1)
    assert st == 0
    assert np.array_equal(got, oracle_mod.fps(pts, m))


# the CTAs of a cluster, a block, and the points a cluster holds (196,608), with neighbours
@pytest.mark.parametrize("n,m", [(1, 1), (2, 2), (15, 15), (16, 16), (17, 9), (33, 33), (255, 200), (4097, 1200),
                                 (32768, 600), (32769, 600), (65537, 300), (196608, 80), (196609, 80)])
def test_sizes(hv, ctx, oracle_mod, n, m):
    check(hv, ctx, oracle_mod, scenes.room_scene(n, seed=n), m)


def grid(a, b, c):
    return np.stack(np.meshgrid(np.arange(a), np.arange(b), np.arange(c), indexing="ij"), -1).reshape(-1, 3)


@pytest.mark.parametrize("form", ["ties", "shuffled ties", "line", "copies", "same", "clusters", "scan", "not finite"])
def test_forms(hv, ctx, oracle_mod, form):
    rng = np.random.default_rng(3)
    box = scenes.uniform_box(3000, 4)
    pts = {"ties": lambda: grid(17, 16, 16),
           "shuffled ties": lambda: rng.permutation(grid(20, 20, 9)),
           "line": lambda: np.outer(np.arange(3000), [1, 0, 0]),
           "copies": lambda: np.concatenate([box[:700]] * 5),
           "same": lambda: np.ones((900, 3)),
           "clusters": lambda: np.concatenate([box * 1e-3, box * 1e-3 + 500, box[:50] * 1e3]),
           "scan": lambda: scenes.lidar_exact(20000, 5),
           "not finite": lambda: np.where(rng.random((3000, 1)) < 0.03, np.array([[np.nan, 1, np.inf]]), box)}[form]()
    check(hv, ctx, oracle_mod, pts, min(len(pts), 900))


def test_every_point(hv, ctx, oracle_mod):
    check(hv, ctx, oracle_mod, scenes.uniform_box(1500, 8), 1500)
