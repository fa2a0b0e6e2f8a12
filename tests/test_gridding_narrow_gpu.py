"""Back-projection with a kernel width whose reciprocal overflows float32: every
weight off the grid points is zero, also in tiles that hold fewer coefficients
than lanes."""
import numpy as np
import pytest

from paper_1905_13408_gb300 import spg, synth

pytestmark = pytest.mark.gpu


def test_width_of_a_denormal():
    n, m = 16, 5
    rng = np.random.default_rng(3)
    X = np.fft.fft2(rng.standard_normal((m, n, n))).astype(np.complex64)
    ctf = rng.uniform(0.5, 1, (m, n, n)).astype(np.float32)
    X[:, 0, 0] = 0
    ctf[:, 0, 0] = 1
    g = spg.Grid(n, kernel="gauss", h=1e-39)
    g.add(synth.random_rotations(m, rng).astype(np.float32), X, ctf)
    N = g.finish()[1].cpu().numpy()
    g.close()
    # k = 0 lies on the origin: its 27 points (19 of them NaN, 0 * infinity, as its
    # weight there is); no other coefficient of a random rotation lies on a point
    near = np.abs(np.fft.fftfreq(n) * n) <= 1
    far = ~(near[:, None, None] & near[None, :, None] & near[None, None, : n // 2 + 1])
    assert (N[far] == 0).all()
