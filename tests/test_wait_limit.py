"""The bounded wait of the tensor-core kernels and of the acceptance runs out (no fault, no hang): the waiter
that reaches its limit gives up, the CTA's other waiters are released, and the status is recorded once."""
import os
import subprocess

import pytest

from paper_2402_02082_gb300 import build

HERE = os.path.dirname(os.path.abspath(__file__))
pytestmark = pytest.mark.gpu


def test_small_wait_runs_out(tmp_path):
    exe = str(tmp_path / "wait_check")
    cmd = [build.nvcc(), *build.ARCH, "-std=c++17", "-O3", "--expt-relaxed-constexpr", "-I", build.CSRC,
           "-I", build.INCLUDE, os.path.join(HERE, "wait_check.cu"), "-o", exe]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr
    r = subprocess.run([exe], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout + r.stderr
    limit, released, warp, done, again, status, *us = (int(x) for x in r.stdout.split())
    assert (limit, released, warp) == (0, 0, 0)  # gave up; nothing else would have ended these waits
    assert (done, again) == (1, 1)
    assert status == 4                           # kStatusTimeout: a wait that ran out
    assert 19000 <= us[0] <= 60000               # the limit of 20 ms
    assert us[1] <= 80000 and us[2] <= 80000     # released by the flag, not by their limits of 2 and 1 s
    assert us[3] <= 5000
