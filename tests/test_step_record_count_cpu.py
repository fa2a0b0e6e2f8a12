"""The count of recorded iterations in a launch of the fused step
(recorded_before, spg_step_kernel.cuh), compiled for the host from the
kernel's source, against counting one by one, for recording intervals up to
the largest an int holds."""
import ctypes
import os
import re
import subprocess

import pytest

from paper_1905_13408_gb300 import build


@pytest.fixture(scope="module")
def recorded_before(tmp_path_factory):
    src = open(os.path.join(build.CSRC, "spg_step_kernel.cuh")).read()
    body = re.search(r"int recorded_before\(.*?\n\}", src, re.S).group(0)
    d = tmp_path_factory.mktemp("rec")
    (d / "rec.cpp").write_text('extern "C" ' + body + "\n")
    subprocess.run(["g++", "-O1", "-fwrapv", "-shared", "-fPIC", "-o", str(d / "rec.so"), str(d / "rec.cpp")], check=True)
    return ctypes.CDLL(str(d / "rec.so")).recorded_before


BIG = 2 ** 31 - 1


@pytest.mark.parametrize("every", [1, 2, 3, 7, 23, 1000, 1 << 30, BIG - 1, BIG])
def test_count(recorded_before, every):
    for rec0 in sorted({r % every for r in (0, 1, 2, 5, every // 2, every - 3, every - 2, every - 1)}):
        for i in (0, 1, 2, 3, 4, 6, 23, 24, 600, 1024):
            assert recorded_before(rec0, every, i) == sum((rec0 + j) % every == 0 for j in range(i)), (rec0, i)


def test_no_recording(recorded_before):
    assert recorded_before(0, 0, 50) == 0
