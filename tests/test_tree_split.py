"""Which kernel takes an fp32 verification over a very long cache (csrc/tree_direct.cu's rule, on the host with
the runtime faked): one or two slabs of a few rows go to the streaming kernel, which spreads the keys over the
chip; more slabs, more rows and shorter caches do not."""
import os
import subprocess

from paper_2402_02082_gb300 import build

HERE = os.path.dirname(os.path.abspath(__file__))


def test_long_caches(tmp_path):
    exe = str(tmp_path / "check")
    cmd = [build.nvcc(), "-gencode", "arch=compute_103a,code=compute_103a", "-std=c++17", "-O0",
           "--expt-relaxed-constexpr", "-I", build.CSRC, "-I", build.INCLUDE, "-I", HERE,
           os.path.join(HERE, "tree_split_check.cu"), "-o", exe]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr
    # B, H, H_kv, D, keys, n, tree
    streaming = [(1, 1, 1, 64, 40000, 1, 1), (1, 1, 1, 64, 65536, 2, 1), (1, 1, 1, 64, 100000, 5, 1),
                 (1, 2, 2, 64, 65536, 1, 1), (2, 1, 1, 64, 100000, 2, 1), (1, 4, 2, 64, 65536, 1, 0),
                 (1, 4, 2, 64, 100000, 2, 1), (1, 1, 1, 128, 65536, 2, 1), (1, 2, 2, 128, 100000, 1, 1),
                 (1, 4, 2, 128, 100000, 1, 0)]
    direct = [(1, 1, 1, 64, 32000, 1, 1), (1, 1, 1, 64, 100000, 9, 1), (1, 4, 4, 64, 100000, 1, 1),
              (2, 4, 4, 64, 65536, 5, 1), (1, 4, 2, 64, 100000, 5, 1), (1, 1, 1, 128, 32000, 5, 1),
              (1, 2, 2, 128, 65536, 9, 1), (1, 4, 2, 128, 100000, 5, 1), (1, 8, 2, 128, 65536, 1, 0),
              (1, 4, 4, 64, 778, 5, 1)]
    lines = "\n".join(" ".join(map(str, s)) for s in streaming + direct)
    r = subprocess.run([exe], input=lines, capture_output=True, text=True, timeout=60)
    got = [int(x) for x in r.stdout.split()]
    assert r.returncode == 0 and len(got) == len(streaming) + len(direct)
    for s, ctas in zip(streaming, got):
        assert ctas == 0, s
    for s, ctas in zip(direct, got[len(streaming):]):
        assert ctas > 0, s
