"""spg_set_data of device arrays (one pass that copies, converts and validates)
against the same arrays handed over from the host (copies, then a validation
pass): stored b and w, seen through a solve, and every verdict are the same."""
import numpy as np
import pytest
import torch

from paper_1905_13408_gb300 import spg, synth

pytestmark = pytest.mark.gpu

HYPER = dict(synth.DEFAULT_HYPER)


def solve(shape, b, w, dtype, storage):
    s = spg.SPG(dict(shape=shape, **HYPER), data_dtype=storage)
    s.set_data(0, b, w, dtype)
    s.reweight()
    s.iterate(3)
    out = s.get_x(0).cpu().numpy(), s.round_stats(0), s.param_scales(0)
    s.close()
    return out


@pytest.mark.parametrize("storage", ["f32", "bf16"])
@pytest.mark.parametrize("src", ["f32", "bf16"])
@pytest.mark.parametrize("shape,offset", [((1, 1, 1), 0), ((5, 9, 128), 0), ((5, 9, 132), 1), ((3, 17, 131), 0),
                                          ((9, 8, 260), 0), ((6, 7, 33), 3)], ids=str)
def test_device_arrays_equal_host_arrays(shape, offset, src, storage):
    n = int(np.prod(shape))
    rng = np.random.default_rng(n)
    t = torch.bfloat16 if src == "bf16" else torch.float32
    dev = []
    for v in (rng.standard_normal(n), np.exp(0.5 * rng.standard_normal(n))):
        buf = torch.zeros(n + offset, dtype=t, device="cuda")
        buf[offset:] = torch.from_numpy(v.astype(np.float32)).cuda().to(t)
        dev.append(buf[offset:].view(shape))  # offset: not on a 16-byte boundary
    dtype = spg.SPG_BF16 if src == "bf16" else spg.SPG_F32
    a = solve(shape, dev[0], dev[1], dtype, storage)
    h = solve(shape, dev[0].cpu(), dev[1].cpu(), dtype, storage)
    np.testing.assert_array_equal(a[0], h[0])
    np.testing.assert_array_equal(a[1], h[1])
    assert a[2] == h[2]


@pytest.mark.parametrize("shape", [(4, 5, 64), (4, 5, 67)], ids=str)
@pytest.mark.parametrize("where,value,status", [("b", np.nan, spg.SPG_ENONFINITE), ("b", np.inf, spg.SPG_ENONFINITE),
                                                ("w", np.nan, spg.SPG_EINVAL), ("w", np.inf, spg.SPG_EINVAL),
                                                ("w", 0.0, spg.SPG_EINVAL), ("w", -1.0, spg.SPG_EINVAL),
                                                ("w", 3.4e38, spg.SPG_EINVAL)])  # rounds to infinity in bfloat16
def test_verdicts(shape, where, value, status):
    b, w = torch.zeros(shape, device="cuda"), torch.ones(shape, device="cuda")
    (b if where == "b" else w)[3, 4, shape[2] - 1] = value
    s = spg.SPG(dict(shape=shape, **HYPER), data_dtype="bf16")
    for bb, ww in ((b, w), (b.cpu(), w.cpu())):
        with pytest.raises(spg.SPGError) as e:
            s.set_data(0, bb, ww)
        assert e.value.status == status
    s.close()
