"""What bench.py says about its kernels: the launches it counts, and which source a recorded DRAM figure is for."""
import os
import shutil

import bench
from paper_2402_02082_gb300 import synth


def test_launches_per_call():
    by_name = {w.name: w for w in synth.workloads()}
    for w in by_name.values():
        for call in ("glide_cross_attn", "tree_accept", "cape_expand", "glide_kv_compact"):
            assert bench.launches_per_call(call, w, False) == 1
        # the split merge is the tensor-core kernels' second launch; fp32 and the CUDA-core kernels have none
        assert bench.launches_per_call("tree_verify_attn", w, False) == (2 if w.dtype == "bf16" else 1)
        assert bench.launches_per_call("tree_verify_attn", w, True) == 1
    assert {w.dtype for w in by_name.values()} == {"bf16", "f32"}


def test_recorded_traffic_follows_the_headers(tmp_path, monkeypatch):
    csrc = os.path.join("paper_2402_02082_gb300", "csrc")
    shutil.copytree(os.path.join(bench.ROOT, csrc), tmp_path / csrc)
    before = {k: bench.kernel_source_hash(f) for k, f in bench.KERNEL_FILES.items()}
    monkeypatch.setattr(bench, "ROOT", str(tmp_path))
    assert before == {k: bench.kernel_source_hash(f) for k, f in bench.KERNEL_FILES.items()}
    with open(tmp_path / csrc / "common.cuh", "a") as f:
        f.write("// changed\n")
    for k, f in bench.KERNEL_FILES.items():
        assert bench.kernel_source_hash(f) != before[k]
