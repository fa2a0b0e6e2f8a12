"""Fourier-domain data term where the GPU has room for the library's transforms
but not for the row pass's own copies of the spectra: the calls succeed on the
library's transforms and give what SPG_ROW_PASS=0 gives."""
import numpy as np
import pytest
import torch

from paper_1905_13408_gb300 import spg, synth

pytestmark = pytest.mark.gpu

SLACK = 24 << 20
BOXES = [(300, 320, 288), (256, 320, 256)]  # both passes of mixed radices; the power-of-two row pass


def free_bytes():
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    return torch.cuda.mem_get_info()[0]


def leave(nbytes):
    """Allocations that leave about nbytes free."""
    held, piece = [], 64 << 30
    while piece >= 2 << 20:
        if free_bytes() - nbytes >= piece:
            held.append(torch.empty(piece, dtype=torch.uint8, device="cuda"))
        else:
            piece //= 2
    return held


class Case:
    def __init__(self, shape):
        g = torch.Generator(device="cuda").manual_seed(5)
        x = torch.rand(shape, generator=g, device="cuda")
        self.shape, self.anchor = shape, 0.5 * x
        self.y = torch.fft.rfftn(x, norm="ortho").contiguous()
        self.N = torch.rand(self.y.shape, generator=g, device="cuda") + 0.1
        self.out = torch.empty(shape, device="cuda")

    def context(self):
        return spg.SPG(dict(shape=self.shape, **dict(synth.DEFAULT_HYPER, mu=0.02)))

    def result(self, s, iters=3):
        s.solve(1, iters)
        x = s.get_x(0, self.out).cpu().numpy().copy()
        return x

    def used(self, anchor):
        """Bytes that set_data_fourier (or the anchor on top) takes, and the result."""
        s = self.context()
        f0 = free_bytes()
        s.set_data_fourier(0, self.y, self.N)
        f1 = free_bytes()
        if anchor:
            s.set_anchor(0, 0.05, self.anchor)
        n0 = s.launch_count()
        x = self.result(s)
        n = s.launch_count() - n0
        f2 = free_bytes()
        s.close()
        return (f1 - f2 if anchor else f0 - f1), x, n


@pytest.mark.parametrize("shape", BOXES, ids=lambda v: "x".join(map(str, v)))
@pytest.mark.parametrize("anchor", [False, True], ids=["data", "anchor"])
def test_row_pass_is_given_up(shape, anchor, monkeypatch):
    c = Case(shape)
    own, x_own, n_own = c.used(anchor)
    monkeypatch.setenv("SPG_ROW_PASS", "0")
    lib, x_lib, n_lib = c.used(anchor)
    monkeypatch.delenv("SPG_ROW_PASS")
    assert own > lib + 4 * SLACK and n_own > n_lib
    # the anchor's share may count memory that the solve takes as well
    for part in (0.35, 0.6, 0.85):
        s = c.context()
        if anchor:
            s.set_data_fourier(0, c.y, c.N)
        held = leave(lib + SLACK + int(part * (own - lib - 2 * SLACK)))
        try:
            if anchor:
                s.set_anchor(0, 0.05, c.anchor)
            else:
                s.set_data_fourier(0, c.y, c.N)
            n0 = s.launch_count()
            x = c.result(s)
            n = s.launch_count() - n0
        finally:
            del held
            torch.cuda.empty_cache()  # the other tests' contexts allocate beside torch's cache
            s.close()
        assert n == n_lib  # the library's transforms
        np.testing.assert_array_equal(x, x_lib)
