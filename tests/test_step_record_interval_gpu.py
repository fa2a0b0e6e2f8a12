"""Objective history at recording intervals near the largest an int holds."""
import pytest

from paper_1905_13408_gb300 import spg, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("every", [1 << 30, 2 ** 31 - 2, 2 ** 31 - 1])
def test_only_the_first_iteration_is_recorded(every):
    shape = (6, 10, 40)
    s = spg.SPG(dict(shape=shape, **synth.DEFAULT_HYPER), hist_every=every)
    s.set_data(0, synth.random_volume(shape, 1).astype("f4"), synth.random_volume(shape, 2, positive=True).astype("f4"))
    s.reweight()
    for k in (1, 5, 1, 7):
        s.iterate(k)
        h = s.history(0)
        assert h.shape[0] == 1 and h[0, 0] == 0
    s.close()
