"""The fused step's barrier over the grid gives up after its limit, and the
context goes on as if nothing had been launched."""
import time

import numpy as np
import pytest

from paper_1905_13408_gb300 import spg, synth

pytestmark = pytest.mark.gpu

HYPER = dict(synth.DEFAULT_HYPER)


@pytest.mark.parametrize("shape,opt", [((4, 5, 9), {}), ((30, 61, 200), dict(storage="prev")),
                                       ((64, 128, 128), dict(data_dtype="bf16", tile="64x4"))],
                         ids=["one-cta", "prev", "many-ctas"])
def test_barrier_gives_up(shape, opt):
    b = synth.random_volume(shape, 3).astype(np.float32)
    w = synth.random_volume(shape, 4, positive=True).astype(np.float32)
    out = []
    for probe in (False, True):
        s = spg.SPG(dict(shape=shape, **HYPER), **opt)
        s.set_data(0, b, w)
        s.reweight()
        s.iterate(7)
        if probe:
            t0 = time.perf_counter()
            assert spg.spg_probe_barrier(s.handle, 20_000_000) == spg.SPG_ETIMEOUT
            assert time.perf_counter() - t0 < 1.0
            assert spg.spg_probe_barrier(s.handle, 1_000_000) == spg.SPG_ETIMEOUT
        s.iterate(9)
        out.append((s.get_x(0).cpu().numpy(), s.history(0), s.counters()))
        s.close()
    np.testing.assert_array_equal(out[0][0], out[1][0])
    np.testing.assert_array_equal(out[0][1], out[1][1])
    assert out[0][2] == out[1][2]


def test_arguments():
    s = spg.SPG(dict(shape=(4, 5, 9), **HYPER))
    for bad in (0, -1, 3_000_000_000):
        assert spg.spg_probe_barrier(s.handle, bad) == spg.SPG_EINVAL
    s.close()
    s = spg.SPG([dict(shape=(4, 5, 9), **HYPER)] * 2)
    assert spg.spg_probe_barrier(s.handle, 1_000_000) == spg.SPG_EINVAL
    s.close()
