"""Back-projection with matrices that are no rotations: positions far outside
the box, which wrap, and weights of positions beyond any index."""
import numpy as np
import pytest

from paper_1905_13408_gb300 import spg, synth
from test_gridding_tiles_gpu import check

pytestmark = pytest.mark.gpu


# the bounds of the tiles' comparison with the oracle; n a power of two, so that
# the oracle's frequencies are exact integers
@pytest.mark.parametrize("kernel", ["gauss", "trilinear"])
@pytest.mark.parametrize("scale", [1e4, 3e5, 4e6])
def test_far_positions(scale, kernel):
    rot = synth.random_rotations(6, np.random.default_rng(int(scale) % 1000))
    check((scale * rot).astype(np.float32), 32, kernel, 2.0, 9)


def test_beyond_int_contributes_nothing():
    """Positions beyond 2^31 have Gaussian weight zero; only k = 0 is left."""
    n, m = 16, 3
    rng = np.random.default_rng(2)
    rot = (1e11 * synth.random_rotations(m, rng)).astype(np.float32)
    X = np.fft.fft2(rng.standard_normal((m, n, n))).astype(np.complex64)
    ctf = rng.uniform(0.5, 1, (m, n, n)).astype(np.float32)
    got = []
    for x in (X, X * (np.add.outer(np.arange(n), np.arange(n)) == 0)):
        g = spg.Grid(n, kernel="gauss")
        c = ctf * (x != 0)
        g.add(rot, x.astype(np.complex64), c.astype(np.float32))
        got.append([t.cpu().numpy() for t in g.finish()])
        g.close()
    # the same up to the order of the sums over images: float64, then float32
    np.testing.assert_allclose(got[0][0], got[1][0], rtol=2.0 ** -22)
    np.testing.assert_allclose(got[0][1], got[1][1], rtol=2.0 ** -22)
