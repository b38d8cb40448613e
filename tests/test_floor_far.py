"""The cell of a point (hav_device.cuh, the counting loops' floor without a
division) from the source itself, built for the host: the floor of the correctly
rounded quotient for boxes up to 2^25 cells from the origin, with the
reciprocal as far off as its intrinsic may be."""
import ctypes as C

import numpy as np
import pytest

import _host_cuda as H

F = np.float32

# A grid over a box as the kernels put it together, an axis at a time, and its points' cells.
CODE = r"""
// out[0]: cells that are not the floor's, out[1]: out of the box, out[2]: taken without a second look
extern "C" int cells(const float* pts, int n, float s, const float* aspect, long long* out) {
    float mn[3], mx[3];
    for (int a = 0; a < 3; ++a) {
        mn[a] = mx[a] = pts[a];
        for (int i = 1; i < n; ++i) mn[a] = fminf(mn[a], pts[3 * i + a]), mx[a] = fmaxf(mx[a], pts[3 * i + a]);
    }
    BoxGrid b;
    unsigned span[3];
    float vmax = 0.0f;
    for (int a = 0; a < 3; ++a) {
        float f0;
        if (!box_axis(s, aspect[a], mn[a], mx[a], &b.g.v[a], &b.ra[a], &f0, &span[a]) || !span[a]) return 0;
        b.g.fmin[a] = f0;
        b.ci[a] = (fabsf(f0) < 4194304.0f) ? -(kMagicBits + static_cast<int>(f0)) : 0;
        vmax = fmaxf(vmax, near_width(b.g.v[a], f0, span[a]));
    }
    b.cells = static_cast<unsigned long long>(span[0]) * span[1] * span[2];
    if (b.cells >= kNoCell) return 0;
    b.amb = __fmul_rn(vmax, kNear);
    b.nx = span[0];
    b.nxy = span[0] * span[1];
    b.c0 = static_cast<unsigned>(b.ci[0]) + b.nx * static_cast<unsigned>(b.ci[1]) + b.nxy * static_cast<unsigned>(b.ci[2]);
    out[0] = out[1] = out[2] = 0;
    const CellMap map(b);
    for (int i = 0; i < n; ++i) {
        const float4 q = {pts[3 * i], pts[3 * i + 1], pts[3 * i + 2], 0.0f};
        const float p[3] = {q.x, q.y, q.z};
        unsigned c = 0, want = 0, stride = 1;
        if (map.fast(q, &c)) ++out[2];
        else c = map.near(q);
        int u[3];
        floor_cells(p, b, u);
        bool same = true;
        for (int a = 0; a < 3; ++a) {
            const float e = floorf(p[a] / b.g.v[a]) - floorf(mn[a] / b.g.v[a]);
            same = same && u[a] == static_cast<int>(e);
            want += stride * static_cast<unsigned>(e);
            stride *= span[a];
        }
        out[0] += (same && c == want) ? 0 : 1;
        out[1] += c < b.cells ? 0 : 1;
    }
    return 1;
}
"""


@pytest.fixture(scope="module", params=[-2, -1, 0, 1, 2], ids=lambda u: f"{u:+d} ulp")
def cells(request, tmp_path_factory):
    text = H.passage("hav_device.cuh", "struct Grid {", "// At most this many voxels are occupied")
    lib = H.compile_host(tmp_path_factory.mktemp("cells"), text + CODE, f"-DULPS={request.param}")

    def run(pts, s, aspect=(1, 1, 1)):
        pts = np.ascontiguousarray(pts, dtype=F)
        out = (C.c_longlong * 3)()
        asp = (C.c_float * 3)(*aspect)
        counted = lib.cells(pts.ctypes.data_as(C.POINTER(C.c_float)), len(pts), C.c_float(s), asp, out)
        return counted, out[0], out[1], out[2] / len(pts)

    return run


def cloud(rng, n, v, base, span):
    """Points of a box that starts `base` cells from the origin, half of them at and beside multiples of v."""
    q = base + rng.uniform(0, 1, (n, 3)) * np.asarray(span)
    q[: n // 2] = np.rint(q[: n // 2])
    x = (q * np.asarray(v, np.float64)).astype(F)
    step = rng.integers(-2, 3, x.shape).astype(np.int32)
    step[n // 2:] = 0
    return np.where(x == 0, x, (x.view(np.int32) + step).view(F))


# cells from the origin: up to 2^20 the fast loop's own, then the division's, to beyond 2^24
@pytest.mark.parametrize("far", [12, 19, 19.9, 20, 20.5, 21, 21.3, 21.9, 22, 22.1, 22.7, 23, 24, 25])
@pytest.mark.parametrize("sign", [1, -1])
def test_far_from_the_origin(cells, far, sign):
    rng = np.random.default_rng(int(100 * far) + sign)
    counted = 0
    for it in range(30):
        s = F(np.exp(rng.uniform(-8, 4)))
        base = np.array([sign * 2.0**far * rng.uniform(1, 1.2), rng.uniform(-300, 300), rng.uniform(-2.0**18, 2.0**18)])
        base = base[rng.permutation(3)]
        pts = cloud(rng, 2000, s, base, rng.choice([3, 40, 900], 3))
        ok, wrong, outside, _ = cells(pts, s)
        counted += ok
        if ok:
            assert wrong == 0 and outside == 0, (far, sign, it)
    assert counted >= 20


# boxes of up to 2^21 cells along an axis, which reach from far to near (or across the origin)
@pytest.mark.parametrize("lo,hi", [(-4194320, -2200000), (-2097152, -10), (-1048580, 1048570), (-1048570, 1048560),
                                   (3, 2097150), (1048000, 3000000), (2200000, 4194330), (-3000, 2000000)])
def test_long_boxes(cells, lo, hi):
    rng = np.random.default_rng(hi & 0xffff)
    for it in range(20):
        s = F(np.exp(rng.uniform(-8, 4)))
        q = cloud(rng, 3000, s, np.array([lo, -5, 7]), np.array([hi - lo, 11, 9]))
        ok, wrong, outside, _ = cells(q[:, rng.permutation(3)], s)
        assert ok and wrong == 0 and outside == 0, it


# anisotropic voxels; near the origin hardly a point takes a second look
@pytest.mark.parametrize("aspect", [(1, 1, 1), (1, 1, 2), (0.1, 1, 3), (8, 0.5, 1)])
def test_near_the_origin(cells, aspect):
    rng = np.random.default_rng(7)
    for it in range(20):
        s = F(np.exp(rng.uniform(-6, 4)))
        v = (s * np.asarray(aspect, dtype=F)).astype(F)
        pts = cloud(rng, 4000, v, rng.uniform(-900, 900, 3), rng.choice([3, 40, 900], 3))
        ok, wrong, outside, fast = cells(pts, s, aspect)
        assert ok and wrong == 0 and outside == 0, it
        fast_only = cells(pts[len(pts) // 2:], s, aspect)[3]  # (the random half)
        assert fast_only > 0.95, (it, fast_only)  # (2 k 2^-22 times the widest voxel over its own, an axis)
