"""Tiles of the back-projection: ragged and partial tiles, boxes that need two
halves or do not fit at all, half-way positions, against the numpy oracle."""
import numpy as np
import pytest

from oracle import gridding
from paper_1905_13408_gb300 import spg, synth

pytestmark = pytest.mark.gpu


def check(rot, n, kernel, h, seed, pw=None):
    rng = np.random.default_rng(seed)
    m = rot.shape[0]
    X = np.fft.fft2(rng.standard_normal((m, n, n))).astype(np.complex64)
    k2 = np.add.outer(np.fft.fftfreq(n) ** 2, np.fft.fftfreq(n) ** 2)
    ctf = np.sin(0.5 + 30.0 * rng.uniform(0.5, 1.5, (m, 1, 1)) * k2).astype(np.float32)
    g = spg.Grid(n, kernel=kernel, h=h)
    g.add(rot, X, ctf, pw)
    y, N = g.finish()
    g.close()
    num, Nf = gridding.grid(X.astype(np.complex128), ctf.astype(np.float64), rot.astype(np.float64), n, kernel, h,
                            pw=None if pw is None else pw.astype(np.float64))
    yr, Nr = gridding.to_fourier_term(num, Nf)
    yr, Nr = synth.half_spectrum(yr), synth.half_spectrum(Nr)
    # float32 weights and tile sums: a few roundings of 2^-24 per deposit
    np.testing.assert_allclose(N.cpu().numpy(), Nr, rtol=1e-6, atol=1e-6 * Nr.max())
    np.testing.assert_allclose(y.cpu().numpy(), yr, rtol=1e-5, atol=2e-6 * np.abs(yr).max())


@pytest.mark.parametrize("kernel", ["gauss", "trilinear"])
@pytest.mark.parametrize("n", [6, 8, 14, 18, 34, 66])
def test_sizes(n, kernel):
    rng = np.random.default_rng(n)
    check(synth.random_rotations(7, rng).astype(np.float32), n, kernel, 2.0, n + 1,
          pw=rng.uniform(0, 1, 7).astype(np.float32))


@pytest.mark.parametrize("kernel", ["gauss", "trilinear"])
def test_half_way_positions(kernel):
    """Axis-aligned planes (every position on a grid point), and columns of
    0.5 and 0.25, whose positions fall on half-way points (a power-of-two n:
    the oracle's frequencies fftfreq(n) * n are then exact integers)."""
    R = [np.eye(3), np.eye(3)[[1, 2, 0]], np.eye(3)[[2, 0, 1]]]
    for a in (0.5, 0.25):
        M = np.zeros((3, 3))
        M[:, 0] = (a, -a, a)
        M[:, 1] = (a, a, -0.5)
        R.append(M)
    check(np.array(R, dtype=np.float32), 32, kernel, 2.0, 5)


def test_other_kernel_width():
    check(synth.random_rotations(5, np.random.default_rng(1)).astype(np.float32), 20, "gauss", 0.7, 6)
