"""The float32-pair evaluation of a coefficient's position (spg_grid.cu,
split_axis), restated in numpy: the nearest-point and floor decisions equal
those of double arithmetic and the remainder is the exact one rounded."""
import numpy as np
import pytest

from paper_1905_13408_gb300 import synth

f32, f64 = np.float32, np.float64


def two_sum(a, b):
    s = a + b
    bb = s - a
    return s, (a - (s - bb)) + (b - bb)


def split_axis(r0, r1, x, y, kernel):
    p, q = (r0 * x).astype(f32), (r1 * y).astype(f32)
    e0 = (r0.astype(f64) * x - p).astype(f32)  # fma(r0, x, -p): exact
    e1 = (r1.astype(f64) * y - q).astype(f32)
    s, t = two_sum(p, q)
    s, lo = two_sum(s, t + (e0 + e1))
    if kernel == 0:
        c = np.rint(s)
        r = (s - c).astype(f32)
        up = ((r - f32(0.5)) + lo).astype(f32) > 0
        dn = ((r + f32(0.5)) + lo).astype(f32) < 0
        c = c + np.where(up, f32(1), np.where(dn, f32(-1), f32(0)))
    else:
        c = np.floor(s)
        c = c - np.where(((s - c) == 0) & (lo < 0), f32(1), f32(0))
    return c.astype(np.int64), ((s - c).astype(f32) + lo).astype(f32)


def grids(n):
    k = np.arange(-n // 2, n // 2)
    ky, kx = np.meshgrid(k[n // 2:], k, indexing="ij")
    return kx.ravel().astype(f32), ky.ravel().astype(f32)


def cases():
    rng = np.random.default_rng(4)
    yield "random", synth.random_rotations(60, rng).astype(f32)[:, :, :2].reshape(-1, 2)
    ties = np.array([0, 0.5, -0.5, 0.25, 1, -1, 0.125, 0.75, 1 / 3, 0.5 + 2.0 ** -24, 0.5 - 2.0 ** -25,
                     2.0 ** -30, -2.0 ** -40, 1e-12], dtype=f32)
    yield "ties", np.array([(a, b) for a in ties for b in ties], dtype=f32)
    near = rng.integers(-8, 8, (200, 2)) * 0.0625 + rng.choice([-1, 0, 1], (200, 2)) * 2.0 ** -27
    yield "near-ties", near.astype(f32)


@pytest.mark.parametrize("kernel", [0, 1])
@pytest.mark.parametrize("name,pairs", list(cases()), ids=lambda v: v if isinstance(v, str) else "")
def test_split_equals_double(name, pairs, kernel):
    x, y = grids(256)
    for r0, r1 in pairs:
        b, f = split_axis(np.full_like(x, r0), np.full_like(y, r1), x, y, kernel)
        p = f64(r0) * x.astype(f64) + f64(r1) * y.astype(f64)
        want = np.rint(p) if kernel == 0 else np.floor(p)
        np.testing.assert_array_equal(b, want.astype(np.int64))
        # one float32 rounding of lo (at most 2^-24 * 2^-17) and one of the sum
        assert np.abs(f.astype(f64) - (p - want)).max() <= 2.0 ** -24
