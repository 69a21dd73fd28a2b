"""Every CTA of the verification kernels looks up its share of the key tiles on its own (build_share in
csrc/common.cuh); the merge finds the shares of a slab by another route (CostPartition).  Both have to agree
tile for tile: tests/share_check.cu runs the library's own code for every share of random batches."""
import os
import subprocess

import pytest

from paper_2402_02082_gb300 import build

HERE = os.path.dirname(os.path.abspath(__file__))
pytestmark = pytest.mark.gpu


def test_shares_agree_with_the_partition(tmp_path):
    exe = str(tmp_path / "share_check")
    cmd = [build.nvcc(), *build.ARCH, "-std=c++17", "-O3", "--expt-relaxed-constexpr", "-I", build.CSRC,
           "-I", build.INCLUDE, os.path.join(HERE, "share_check.cu"), "-o", exe]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr
    r = subprocess.run([exe], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0 and r.stdout.startswith("ok"), r.stdout + r.stderr
