"""The objective recorded by a launch's last iteration: its sums are read by
CTAs that did not form them, so they have to be stored before the barrier over
the grid. Launches of two iterations against launches of one, whose sums are
read by the last CTA to finish; the entries are bitwise the same."""
import numpy as np
import pytest

from paper_1905_13408_gb300 import spg, synth

pytestmark = pytest.mark.gpu

HYPER = dict(synth.DEFAULT_HYPER)


# weights spread over 10^5, so that the objective keeps falling; at 1e30 the
# sums take the longer double branch
@pytest.mark.parametrize("wscale", [1.0, 1e30], ids=["ordinary", "above-float32"])
@pytest.mark.parametrize("shapes,opt", [
    ([(24, 40, 128)], dict(tile="128x7s4", zchunk=1)),
    ([(40, 61, 200)], dict(tile="64x4", zchunk=3)),
    ([(16, 45, 150)], dict(tile="128x15", storage="prev")),
    ([(12, 20, 64), (9, 31, 130), (30, 14, 40)], dict(data_dtype="bf16")),
], ids=["128x7", "64x4", "128x15", "batch"])
def test_last_entry_of_a_launch(shapes, opt, wscale):
    hists = []
    for chunks in ([2] * 40, [1] * 80):
        s = spg.SPG([dict(shape=sh, **HYPER) for sh in shapes], **opt)
        for j, sh in enumerate(shapes):
            rng = np.random.default_rng(17 + j)
            b = (rng.uniform(500, 1000, sh) * np.sign(rng.standard_normal(sh))).astype(np.float32)
            w = (wscale * 10.0 ** rng.uniform(-5, 0, sh)).astype(np.float32)
            s.set_data(j, b, w)
        s.reweight()
        n0 = s.launch_count()
        for c in chunks:
            s.iterate(c)
        assert s.launch_count() - n0 == len(chunks)
        hists.append([s.history(j) for j in range(len(shapes))])
        s.close()
    for a, b in zip(*hists):
        assert a.shape[0] == 80 and len(set(a[:, 1])) == 80  # no two entries alike: a stale one would show
        np.testing.assert_array_equal(a, b)
