"""Tiles of the back-projection whose box does not fit even in halves (deposited
directly) and boxes longer than the grid (every point wrapped on its own), which
only matrices that are no rotations reach, against the numpy oracle."""
import numpy as np
import pytest

from paper_1905_13408_gb300 import synth
from test_gridding_tiles_gpu import check

pytestmark = pytest.mark.gpu

CAP = 768


def routes(rot, n, kernel):
    """(passes deposited directly, boxes longer than n) of the kernel's tiles of 8 x 4 coefficients."""
    direct = long = 0
    span = 3 if kernel == "gauss" else 2
    for R in rot.astype(np.float64):
        for ky0 in range(0, n // 2, 4):
            for kx0 in range(-n // 2, n // 2, 8):
                k = [(i, x, y) for i, (y, x) in enumerate((y, x) for y in range(ky0, ky0 + 4) for x in range(kx0, kx0 + 8))
                     if x < n // 2 and y < n // 2 and (y > 0 or x > 0) and x * x + y * y <= (n / 2 - 2) ** 2]

                def extents(ks):
                    p = np.array([R[:, 0] * x + R[:, 1] * y for _, x, y in ks])
                    p = np.rint(p) if kernel == "gauss" else np.floor(p)
                    return np.ptp(p, axis=0) + span

                halves = [k] if k and np.prod(extents(k)) <= CAP else [[s for s in k if (s[0] < 16) == h] for h in (True, False)]
                for ks in halves:
                    if not ks:
                        continue
                    e = extents(ks)
                    direct += np.prod(e) > CAP
                    long += np.prod(e) <= CAP and e.max() > n
    return direct, long


@pytest.mark.parametrize("kernel", ["gauss", "trilinear"])
@pytest.mark.parametrize("scale", [4.0, 8.0])
def test_boxes_that_do_not_fit(scale, kernel):
    rot = (scale * synth.random_rotations(6, np.random.default_rng(31))).astype(np.float32)
    assert routes(rot, 32, kernel)[0] > 10
    check(rot, 32, kernel, 2.0, 12, pw=np.random.default_rng(5).uniform(0, 1, 6).astype(np.float32))


@pytest.mark.parametrize("kernel", ["gauss", "trilinear"])
@pytest.mark.parametrize("n,scale", [(8, 8.0), (16, 5.5)])
@pytest.mark.parametrize("axis", [0, 1, 2])
def test_boxes_longer_than_the_grid(axis, n, scale, kernel):
    tilt = np.array([[0.995, -0.08, 0.06], [0.07, 0.99, 0.1], [-0.05, 0.09, 0.99]])
    rot = np.roll(np.diag([scale, 1.0, 1.0]) @ tilt, axis, axis=0)[None].astype(np.float32)
    assert routes(rot, n, kernel)[1] > 0
    check(rot, n, kernel, 2.0, 13)
