"""Farthest point sampling of few points, picked one per barrier: on both sides
of the line to the many-picks form and of the cluster's largest cloud, the
oracle's sequence of picks."""
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


def line(n):
    return min(n // 48, 44 + n // 2048)


@pytest.mark.parametrize("n", [96, 700, 1000, 4096, 16384, 32767, 32768, 32769, 100000, 196608, 196609])
def test_both_sides_of_the_line(hv, ctx, oracle_mod, n):
    pts = scenes.room_scene(n, seed=n)
    for m in sorted({1, 2, max(1, line(n) - 1), line(n), line(n) + 1}):
        check(hv, ctx, oracle_mod, pts, m)


@pytest.mark.parametrize("form", ["ties", "copies", "same", "not finite"])
def test_forms(hv, ctx, oracle_mod, form):
    rng = np.random.default_rng(3)
    box = scenes.uniform_box(8000, 4)
    pts = {"ties": lambda: rng.permutation(
               np.stack(np.meshgrid(*[np.arange(20)] * 3, indexing="ij"), -1).reshape(-1, 3)),
           "copies": lambda: np.concatenate([box[:800]] * 10),
           "same": lambda: np.ones((8000, 3)),
           "not finite": lambda: np.where(rng.random((8000, 1)) < 0.002, np.array([[np.nan, 1, np.inf]]), box)}[form]()
    check(hv, ctx, oracle_mod, pts, line(8000) - 1)


# tied distances first, distinct ones after them (and mixed): the threshold's distance comes back from 0
@pytest.mark.parametrize("form", ["half rounded", "lattice, then a box", "a fine box in a lattice"])
def test_ties_and_distinct_distances(hv, ctx, oracle_mod, form):
    rng = np.random.default_rng(5)
    box = scenes.uniform_box(9000, 6)
    grid = np.stack(np.meshgrid(*[np.arange(16)] * 3, indexing="ij"), -1).reshape(-1, 3)
    pts = {"half rounded": lambda: rng.permutation(np.concatenate([np.rint(box[:4000]), box[4000:8000]])),
           "lattice, then a box": lambda: np.concatenate([grid * 30.0, box[:4000]]),
           "a fine box in a lattice": lambda: np.concatenate([grid * 1.0, box[:4000] * 0.2])}[form]()
    check(hv, ctx, oracle_mod, pts, 2500)
