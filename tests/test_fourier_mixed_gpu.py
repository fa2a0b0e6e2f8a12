"""Mixed-radix passes of the Fourier-domain data term against the library's
transforms (SPG_ROW_PASS=0 when the data are set) on the same solve."""
import numpy as np
import pytest
import torch  # noqa: F401

from paper_1905_13408_gb300 import spg, synth

pytestmark = pytest.mark.gpu


def solve(fv, hyper, iters, anchor=None):
    s = spg.SPG(dict(shape=fv.phantom.shape, **hyper))
    s.set_data_fourier(0, synth.half_spectrum(fv.y).astype(np.complex64), synth.half_spectrum(fv.N).astype(np.float32))
    if anchor is not None:
        s.set_anchor(0, 0.05, anchor)
    s.solve(1, iters)
    x, h = s.get_x(0).cpu().numpy().astype(np.float64), s.history(0)
    n = s.launch_count()
    s.close()
    return x, h, n


# shortest and longest axes of the passes (16 and 512); radices 2 .. 13; odd nx;
# odd ny (row pairs across planes) and ragged groups of rows; ragged tiles along
# z; power-of-two nz, whose pass along z is another, with and without its TMA
# form; all of at least 2^21 coefficients, from which these passes are taken.
# The transforms' roundings (about 3e-7 relative each) meet the same solve as in
# the power-of-two row pass's comparison: its bound, 1e-6.
@pytest.mark.parametrize("shape", [(18, 512, 512), (500, 17, 512), (512, 486, 16), (455, 143, 65), (143, 121, 243),
                                   (182, 182, 126), (128, 330, 100), (256, 256, 64), (392, 99, 110), (180, 180, 180)])
def test_mixed_passes_equal_library_transforms(shape, monkeypatch):
    fv = synth.make_fourier_volume(shape, blobs=12, radius=min(shape) / 3, seed=sum(shape) + 3)
    hyper = dict(synth.DEFAULT_HYPER, mu=0.02)
    x_own, h_own, n_own = solve(fv, hyper, 20)
    monkeypatch.setenv("SPG_ROW_PASS", "0")
    x_lib, h_lib, n_lib = solve(fv, hyper, 20)
    assert n_own > n_lib  # the passes are this library's
    err = float(np.linalg.norm(x_own - x_lib) / np.linalg.norm(x_lib))
    print(f"mixed passes vs library transforms {shape}: rel-L2 {err:.3e}")
    assert err <= 1e-6
    np.testing.assert_allclose(h_own[:, 2:4], h_lib[:, 2:4], rtol=1e-6)


@pytest.mark.parametrize("shape", [(182, 182, 126), (128, 330, 100)])
def test_anchor_on_mixed_passes(shape, monkeypatch):
    """The anchor's N and C in the order of these passes, with either pass along z."""
    fv = synth.make_fourier_volume(shape, blobs=12, radius=min(shape) / 3, seed=sum(shape) + 4)
    hyper = dict(synth.DEFAULT_HYPER, mu=0.02)
    anchor = 0.5 * fv.phantom.astype(np.float32)
    x_own, _, _ = solve(fv, hyper, 20, anchor)
    monkeypatch.setenv("SPG_ROW_PASS", "0")
    x_lib, _, _ = solve(fv, hyper, 20, anchor)
    assert float(np.linalg.norm(x_own - x_lib) / np.linalg.norm(x_lib)) <= 1e-6
