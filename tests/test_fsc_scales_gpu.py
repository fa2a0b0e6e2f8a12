"""FSC of two maps of different scale: the correlation does not change with a
power of two in one map, whichever kernel sums the shells."""
import numpy as np
import pytest
import torch

from paper_1905_13408_gb300 import spg

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("which", [0, 1])
@pytest.mark.parametrize("power", [-100, -82, -74, -66, -50, -20, 45, 70])
def test_one_map_scaled(power, which):
    """Components of the scaled map from 1e-28 to 1e23, the other map's near 200.
    A power of two is exact in the transforms and in the shell sums, but for
    the sums' own rounding (48 bits at least)."""
    rng = np.random.default_rng(8)
    a = rng.standard_normal((40, 40, 40)).astype(np.float32)
    b = (a + 0.7 * rng.standard_normal(a.shape)).astype(np.float32)
    maps = [torch.from_numpy(a).cuda(), torch.from_numpy(b).cuda()]
    want, cnt = spg.spg_fsc(*maps)
    maps[which] = maps[which] * np.float32(2.0 ** power)
    got, cnt2 = spg.spg_fsc(*maps)
    np.testing.assert_array_equal(cnt, cnt2)
    np.testing.assert_allclose(got, want, rtol=0, atol=1e-12)
