"""The partial sums of the NPT step (rbe_npt_plan.h): room for the blocks of each pair kernel and of the finishing
kernel at every particle count, in particular at the small ones where the FP64 pair kernels have more blocks."""
import os
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.mark.parametrize("sms", [1, 148, 152])
@pytest.mark.parametrize("lo,hi", [(1, 6000), (19990, 20010)])
def test_partial_rows_cover_every_block(tmp_path, sms, lo, hi):
    exe = str(tmp_path / "npt_plan")
    subprocess.run(["g++", "-std=c++17", "-O1", "-o", exe, os.path.join(HERE, "host", "npt_plan_main.cpp")], check=True)
    out = subprocess.run([exe, str(sms), str(lo), str(hi)], capture_output=True, text=True, check=True).stdout
    t = np.array([line.split() for line in out.splitlines()], dtype=np.int64)
    assert t.shape == (hi - lo + 1, 6)
    assert np.all(t[:, 5] >= t[:, 1:4].max(1) + t[:, 4])
    assert np.all(t[:, 5] <= 5 * sms + t[:, 4])
