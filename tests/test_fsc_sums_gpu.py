"""Shell sums of the FSC: edges of the lane and index layout, values outside
the float-float range, and where the maps may live."""
import numpy as np
import pytest
import torch

from oracle import fsc as ofsc
from paper_1905_13408_gb300 import spg

pytestmark = pytest.mark.gpu


def maps(n, seed=3):
    rng = np.random.default_rng(seed)
    a = rng.standard_normal((n, n, n)).astype(np.float32)
    return a, (a + 0.7 * rng.standard_normal((n, n, n))).astype(np.float32)


@pytest.mark.parametrize("n", [2, 3, 4, 5, 31, 62, 63, 66, 127, 130])
def test_sizes(n):
    """Lines of one warp, its edges, odd and even (Nyquist) lengths; the
    tolerance is that of the float32 transforms."""
    a, b = maps(n)
    got, cnt = spg.spg_fsc(torch.from_numpy(a).cuda(), torch.from_numpy(b).cuda())
    want, wcnt = ofsc.fsc(a, b)
    np.testing.assert_array_equal(cnt, wcnt)
    np.testing.assert_allclose(got, want, rtol=1e-5, atol=1e-6)


@pytest.mark.parametrize("power", [-60, 60])
def test_scale(power):
    """A power of two in both maps moves every product out of the float-float
    range and changes nothing else: double sums of the same products."""
    a, b = maps(48)
    f0, c0 = spg.spg_fsc(torch.from_numpy(a).cuda(), torch.from_numpy(b).cuda())
    f1, c1 = spg.spg_fsc(torch.from_numpy(a * np.float32(2.0 ** power)).cuda(),
                         torch.from_numpy(b * np.float32(2.0 ** power)).cuda())
    np.testing.assert_array_equal(c0, c1)
    np.testing.assert_allclose(f0, f1, rtol=0, atol=1e-12)


def test_nan_and_zero_maps():
    a, b = maps(20)
    z = torch.zeros(20, 20, 20, device="cuda")
    assert np.isnan(spg.spg_fsc(z, torch.from_numpy(b).cuda())[0]).all()
    a[3, 4, 5] = np.nan
    assert np.isnan(spg.spg_fsc(torch.from_numpy(a).cuda(), torch.from_numpy(b).cuda())[0]).all()


def test_where_the_maps_live():
    """Aligned device maps are transformed in place of a copy and left as they
    were; views at an odd offset, host arrays and calls on another stream give
    the same values."""
    n = 40
    a, b = maps(n)
    da, db = torch.from_numpy(a).cuda(), torch.from_numpy(b).cuda()
    want, _ = spg.spg_fsc(da, db)
    np.testing.assert_array_equal(da.cpu().numpy(), a)
    np.testing.assert_array_equal(db.cpu().numpy(), b)
    buf = torch.empty(n ** 3 + 1, device="cuda")
    view = buf[1:].view(n, n, n)
    view.copy_(da)
    np.testing.assert_array_equal(spg.spg_fsc(view, db)[0], want)
    np.testing.assert_array_equal(spg.spg_fsc(a, b)[0], want)
    side = torch.cuda.Stream()
    torch.cuda.synchronize()
    np.testing.assert_array_equal(spg.spg_fsc(da, db, stream=side.cuda_stream)[0], want)
    with torch.cuda.stream(side):
        np.testing.assert_array_equal(spg.spg_fsc(da, db)[0], want)
    for m in (2, 6, 10, 14, 18, 22):  # more plans than stay idle
        spg.spg_fsc(a[:m, :m, :m].copy(), b[:m, :m, :m].copy())
    np.testing.assert_array_equal(spg.spg_fsc(da, db)[0], want)
