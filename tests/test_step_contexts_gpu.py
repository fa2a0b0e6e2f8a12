"""Contexts beside one another: a launch of the fused step is bounded in time,
so that other contexts' kernels get their turn, and contexts iterating from
several threads on streams of different priority give what each gives alone
(their launches keep every CTA resident and wait across the grid)."""
import threading

import numpy as np
import pytest
import torch

from paper_1905_13408_gb300 import spg, synth

pytestmark = pytest.mark.gpu

HYPER = dict(synth.DEFAULT_HYPER)


def test_launches_are_bounded_in_time():
    """An iteration at 256^3 moves 0.54 GB, 80 us or so: 100 take 8 ms, four launches of 2 ms at least."""
    shape = (256, 256, 256)
    g = torch.Generator(device="cuda").manual_seed(1)
    s = spg.SPG(dict(shape=shape, **HYPER))
    s.set_data(0, torch.rand(shape, generator=g, device="cuda"), 0.5 + torch.rand(shape, generator=g, device="cuda"))
    s.reweight()
    n0 = s.launch_count()
    s.iterate(100)
    launches = s.launch_count() - n0
    s.objective(0)
    s.close()
    assert 4 <= launches <= 10


SHAPES = [(64, 64, 64), (40, 90, 300), (101, 147, 183), (28, 32, 40)]


def solve(j, stream, rounds=6, iters=150):
    shape = SHAPES[j]
    with torch.cuda.stream(stream):
        s = spg.SPG(dict(shape=shape, **HYPER), stream=stream.cuda_stream, restart=j == 1, storage="prev" if j == 3 else "delta")
        s.set_data(0, synth.random_volume(shape, 5 + j).astype(np.float32),
                   synth.random_volume(shape, 50 + j, positive=True).astype(np.float32))
        s.solve(rounds, iters)
        out = s.get_x(0).cpu().numpy(), s.history(0), s.objective(0)
        s.close()
    return out


@pytest.mark.parametrize("priorities", [(0, 0, 0, 0), (-1, 0, 0, -1)], ids=["equal", "mixed"])
def test_contexts_in_several_threads(priorities):
    alone = [solve(j, torch.cuda.Stream()) for j in range(4)]
    got = [None] * 4

    def work(j, stream):
        try:
            got[j] = solve(j, stream)
        except Exception as e:  # e.g. SPG_ETIMEOUT
            got[j] = e

    ts = [threading.Thread(target=work, args=(j, torch.cuda.Stream(priority=p))) for j, p in enumerate(priorities)]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    for a, b in zip(alone, got):
        assert not isinstance(b, Exception), b
        np.testing.assert_array_equal(a[0], b[0])
        np.testing.assert_array_equal(a[1], b[1])
        np.testing.assert_array_equal(a[2], b[2])
