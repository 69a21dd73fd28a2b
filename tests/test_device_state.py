"""What the launchers keep between calls (shared-memory limits, the SM count, the room for clusters)
belongs to a device: host-side, with the runtime faked (tests/fake_cudart.cuh), no GPU."""
import os
import subprocess

import pytest

from paper_2402_02082_gb300 import build

HERE = os.path.dirname(os.path.abspath(__file__))
UNITS = ["device.h", "cross_attn.cu", "tree_attn_fma.cu", "tree_attn_tc.cu", "tree_attn_wide.cu", "block_attn.cu",
         "accept.cu", "sampling.cu"]


@pytest.mark.parametrize("unit", UNITS)
def test_state_is_per_device(unit, tmp_path):
    exe = str(tmp_path / "check")
    # PTX only: nothing of the device code runs
    cmd = [build.nvcc(), "-gencode", "arch=compute_103a,code=compute_103a", "-std=c++17", "-O0",
           "--expt-relaxed-constexpr", "-I", build.CSRC, "-I", build.INCLUDE, "-I", HERE, f'-DUNIT="{unit}"',
           f"-DLAUNCH={UNITS.index(unit)}", os.path.join(HERE, "device_state_check.cu"),
           "-o", exe]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr
    r = subprocess.run([exe], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0 and r.stdout.strip() == "ok", r.stdout + r.stderr
