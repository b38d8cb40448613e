"""The division-free floor of the counting loops (hav_device.cuh, floor_bits and
floor_near) restated in numpy binary32 against floor of the correctly rounded
quotient: random points, points at and beside multiples of v, powers of two,
tiny coordinates, and quotients up to 2^22."""
import numpy as np
import pytest

F = np.float32
MAGIC = F(12582912.0)


def fma(a, b, c):
    # the product of two binary32 numbers is exact in longdouble (64 bits), and so is the sum here
    return (a.astype(np.longdouble) * b.astype(np.longdouble) + c.astype(np.longdouble)).astype(F)


def fast_floor(x, v, amb):
    r = F(1) / v
    s = fma(x, r, np.full_like(x, MAGIC))
    k = s - MAGIC
    rem = fma(-k, v, x)
    away = np.abs(rem) > fma(np.abs(k), amb, amb * F(2.0**-70))
    t = s.view(np.int32) + (rem.view(np.int32) >> 31) - 0x4B400000
    kb = k.view(np.int32)
    p = (np.where(k > 0, kb - 1, kb) & 0x7F800000).astype(np.int32).view(F)
    near = np.where(rem >= -(v * (p * F(2.0**-24))), k, k - F(1))
    div = ~(np.abs(k) < 4194304) | ((k == 0) & (np.abs(x) <= v * F(1e-30)) & (x != 0))
    near = np.where(div, np.floor(x / v), near)
    return np.where(away, t.astype(np.float64), near.astype(np.float64))


@pytest.mark.skipif(np.finfo(np.longdouble).nmant < 63, reason="needs a 64-bit significand")
@pytest.mark.parametrize("form", ["random", "multiples", "powers", "tiny", "large"])
@pytest.mark.parametrize("wider", [1.0, 3.0])
def test_floor_of_the_correctly_rounded_quotient(form, wider):
    rng = np.random.default_rng(5)
    n = 200_000
    for it in range(4):
        v = np.exp(rng.uniform(-12, 6, n)).astype(F) if it % 2 else np.full(n, np.exp(rng.uniform(-8, 4)), F)
        if form == "random":
            x = (rng.uniform(-1, 1, n) * np.exp(rng.uniform(-3, 14, n)) * v).astype(F)
        elif form == "tiny":
            x = (rng.uniform(-1, 1, n) * np.exp(rng.uniform(-100, -60, n))).astype(F)
            x[::7] = 0
            x[::11] = F(-1e-45)
        else:
            k = {"multiples": lambda: rng.integers(-2000, 2000, n),
                 "powers": lambda: 2.0**rng.integers(0, 21, n) * rng.choice([-1, 1], n),
                 "large": lambda: rng.integers(-2**22, 2**22, n)}[form]()
            x = (k * v.astype(np.float64)).astype(F)
            x = (x.view(np.int32) + rng.integers(-3, 4, n).astype(np.int32)).view(F)
        ok = np.isfinite(x) & (np.abs(x) < 1e30)
        x, v = x[ok], v[ok]
        amb = v * F(2.0**-22) * F(wider)  # (2^-22 times the largest v of the three axes)
        assert np.array_equal(fast_floor(x, v, amb), np.floor(x / v).astype(np.float64))
