"""Several iterations in one launch of the fused step against one launch per
iteration: the iterate, the objective history, the counters and the
extrapolation (through the iterations that follow) are bitwise the same."""
import numpy as np
import pytest

from paper_1905_13408_gb300 import spg, synth

pytestmark = pytest.mark.gpu

HYPER = dict(synth.DEFAULT_HYPER)


def run(shapes, chunks, **opt):
    s = spg.SPG([dict(shape=sh, **HYPER) for sh in shapes], **opt)
    for j, sh in enumerate(shapes):
        s.set_data(j, synth.random_volume(sh, 70 + j).astype(np.float32),
                   synth.random_volume(sh, 170 + j, positive=True).astype(np.float32))
    launches = []
    for _ in range(2):
        s.reweight()
        for c in chunks:
            n0 = s.launch_count()
            s.iterate(c)
            launches.append(s.launch_count() - n0)
    out = [(s.get_x(j).cpu().numpy(), s.history(j)) for j in range(len(shapes))]
    state = s.get_state()
    counters = s.counters()
    s.close()
    return out, state, counters, launches


@pytest.mark.parametrize("shapes,opt", [
    ([(1, 1, 1)], {}),
    ([(3, 5, 7)], dict(storage="prev")),
    ([(12, 40, 50)], dict(hist_every=3)),
    ([(33, 61, 200)], dict(tile="64x7", zchunk=4, ctas_per_sm=1)),                   # several items per CTA
    ([(33, 61, 200)], dict(tile="128x15", zchunk=1, ctas_per_sm=1, restart=True)),   # items of 3 plane steps
    ([(20, 30, 64)], dict(restart=True, storage="prev", hist_every=2)),
    ([(9, 17, 33)], dict(hist_capacity=4)),                                          # ring shorter than a launch
    ([(10, 12, 40), (24, 31, 130), (7, 50, 65)], dict(restart=True)),
    ([(10, 12, 40), (24, 31, 130), (7, 50, 65)], dict(data_dtype="bf16", tile="128x4")),
    ([(128, 128, 192)], dict(tile="64x4", zchunk=1, ctas_per_sm=1, restart=True)),   # above kMaxCtaItems: one per launch
], ids=lambda v: "x".join(map(str, v[0])) if isinstance(v, list) else None)
def test_one_launch_equals_single_iterations(shapes, opt):
    n = 6 if shapes[0][0] > 100 else 23
    a = run(shapes, [n], **opt)
    b = run(shapes, [1] * n, **opt)
    for (xa, ha), (xb, hb) in zip(a[0], b[0]):
        np.testing.assert_array_equal(xa, xb)
        np.testing.assert_array_equal(ha, hb)
    assert a[1] == b[1]
    assert a[2] == b[2]
    if shapes[0][0] <= 100:
        assert a[3] == [1, 1]
