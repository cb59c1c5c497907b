"""bench.py's hash of a kernel's sources covers every file the kernel is
compiled from, so that a profile of older sources is not taken for a current
one.  CPU only."""
import glob
import os
import re
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)
CSRC = os.path.join(ROOT, "paper_2601_16791_gb300", "csrc")


def test_kernel_sources_follow_the_includes():
    import bench
    have = {os.path.basename(f) for f in glob.glob(os.path.join(CSRC, "*"))}
    for kernel, files in bench.KERNEL_SOURCES.items():
        for f in files:
            text = open(os.path.join(CSRC, f)).read()
            for inc in re.findall(r'#include\s+"([^"]+)"', text):
                if inc in have:
                    assert inc in files, (kernel, f, inc)
    # the functions these two run besides their own files'
    assert {"mx_split_gas.cuh", "mx_kepler_short.cuh", "mx_bs2.cuh"} <= set(bench.KERNEL_SOURCES["k_catchup"])
    assert "mx_split.cuh" in bench.KERNEL_SOURCES["k_jump_drift"]
