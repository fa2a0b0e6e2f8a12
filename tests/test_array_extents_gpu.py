"""Device arrays shorter than what a call reads are refused on the host (a kernel
or a transform that reads them in place would leave the allocation), and arrays
mapped in pieces are still taken."""
import os
import subprocess
import sys

import numpy as np
import pytest
import torch

from paper_1905_13408_gb300 import spg, synth

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
N = 160  # 16 MB of float32, 8 MB of bfloat16: more than the segment of a small tensor
SHAPE = (N, N, N)


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("short", ["b", "w"])
def test_set_data_refuses_short_arrays(short, dtype):
    tt, code = (torch.float32, spg.SPG_F32) if dtype == "f32" else (torch.bfloat16, spg.SPG_BF16)
    full = torch.rand(SHAPE, device="cuda").to(tt) + 0.5
    torch.cuda.empty_cache()
    small = torch.ones(1000, device="cuda", dtype=tt)
    s = spg.SPG(dict(shape=SHAPE, **synth.DEFAULT_HYPER))
    with pytest.raises(spg.SPGError) as e:
        s.set_data(0, small if short == "b" else full, small if short == "w" else full, code)
    assert e.value.status == spg.SPG_EINVAL and "shorter" in str(e.value)
    s.set_data(0, full, full, code)  # the context goes on
    s.reweight()
    s.iterate(1)
    # x_0 = 0: F = 1/2 sum w b^2; float32 terms (3 roundings, 2^-22)
    want = 0.5 * float((full.double() ** 3).sum())
    assert abs(s.history(0)[0, 1] - want) <= 2.0 ** -22 * want
    s.close()


@pytest.mark.parametrize("short", [0, 1])
def test_fsc_refuses_short_maps(short):
    maps = [torch.rand(SHAPE, device="cuda") for _ in range(2)]
    want = spg.spg_fsc(*maps)[0]
    torch.cuda.empty_cache()
    bad = list(maps)
    bad[short] = torch.ones(N, 2, 2, device="cuda")
    with pytest.raises(spg.SPGError) as e:
        spg.spg_fsc(*bad)
    assert e.value.status == spg.SPG_EINVAL and "shorter" in str(e.value)
    np.testing.assert_array_equal(spg.spg_fsc(*maps)[0], want)


PIECES = """
import numpy as np, torch
from paper_1905_13408_gb300 import spg, synth
shape = (192, 192, 192)
g = torch.Generator(device="cuda").manual_seed(1)
b, w = torch.rand(shape, generator=g, device="cuda"), torch.rand(shape, generator=g, device="cuda") + 0.5
h = b.cpu(), w.cpu()
got = []
for x, y in ((b, w), h):
    s = spg.SPG(dict(shape=shape, **synth.DEFAULT_HYPER))
    s.set_data(0, x, y)
    s.solve(1, 5)
    got.append(s.get_x(0).cpu().numpy())
    s.close()
np.testing.assert_array_equal(*got)
np.testing.assert_array_equal(spg.spg_fsc(b, w)[0], spg.spg_fsc(*h)[0])
print("pieces ok")
"""


def test_arrays_mapped_in_pieces():
    """28 MB arrays in torch's expandable segments, which map memory 20 MB at a time."""
    env = dict(os.environ, PYTORCH_CUDA_ALLOC_CONF="expandable_segments:True", PYTORCH_ALLOC_CONF="expandable_segments:True")
    r = subprocess.run([sys.executable, "-c", PIECES], cwd=ROOT, env=env, capture_output=True, text=True, timeout=600)
    assert r.returncode == 0 and "pieces ok" in r.stdout, (r.stdout + r.stderr)[-2000:]
