"""A captured DRAM figure is valid for the sources it was captured on, headers included."""
import os
import shutil
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)


def test_source_hash_covers_the_headers(tmp_path):
    import bench
    csrc = str(tmp_path / "csrc")
    shutil.copytree(os.path.join(ROOT, "paper_2509_18497_gb300", "csrc"), csrc, ignore=shutil.ignore_patterns("*.o"))
    before = bench._src_sha("rgs_trace.cu", csrc)
    assert before == bench._src_sha("rgs_trace.cu")
    for name in ("rgs_trace.cu", "rgs_warp_trace.cuh", "rgs_internal.cuh"):
        with open(os.path.join(csrc, name), "a") as f:
            f.write("\n")
        after = bench._src_sha("rgs_trace.cu", csrc)
        assert after != before, name
        before = after
