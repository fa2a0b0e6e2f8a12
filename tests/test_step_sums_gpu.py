"""The fused step's objective sums across a CTA: float-float sums, double where
those could overflow, against a float64 evaluation of F(x_0)."""
import numpy as np
import pytest
import torch

from paper_1905_13408_gb300 import spg, synth

pytestmark = pytest.mark.gpu

HYPER = dict(synth.DEFAULT_HYPER)


@pytest.mark.parametrize("wscale", [1.0, 1e30], ids=["ordinary", "above-float32"])
@pytest.mark.parametrize("tile", ["128x7s4", "64x4", "128x8", "128x15"])
def test_first_history_entry(tile, wscale):
    """x_0 = 0: F is the data term 1/2 sum w b^2 alone. With w = 1e30 and
    |b| up to 1000 the terms reach 1e36 and the volume's sum 1e39, which a
    float32 pair cannot hold; each term is one float32 expression (3 roundings,
    2^-22), the sums add far less."""
    shape = (8, 19, 150)
    rng = np.random.default_rng(11)
    b = (rng.uniform(500, 1000, shape) * np.sign(rng.standard_normal(shape))).astype(np.float32)
    w = (wscale * rng.uniform(0.5, 1.0, shape)).astype(np.float32)
    s = spg.SPG(dict(shape=shape, **HYPER), tile=tile)
    s.set_data(0, b, w)
    s.reweight()
    s.iterate(1)
    h = s.history(0)
    s.close()
    want = 0.5 * float((w.astype(np.float64) * b.astype(np.float64) ** 2).sum())
    assert h.shape[0] == 1 and h[0, 0] == 0
    assert abs(h[0, 1] - want) <= 2.0 ** -22 * want
    assert h[0, 2] == 0 and h[0, 3] == 0 and h[0, 4] == h[0, 1]
