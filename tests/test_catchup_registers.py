"""The catch-up kernel's chains set the time of a long run's windows: it is
compiled without spills, for two blocks of 128 threads an SM.  CPU only (the
compiler's own report)."""
import os
import re
import subprocess

import pytest

from paper_2601_16791_gb300 import build


def test_catchup_does_not_spill(tmp_path):
    try:
        nvcc = build._nvcc()
    except RuntimeError:
        pytest.skip("no nvcc")
    r = subprocess.run([nvcc, "-c", os.path.join(build.CSRC, "k_bs.cu"), "-o", str(tmp_path / "k_bs.o")] + build.ARCH +
                       ["-O3", "-std=c++17", "-Xcompiler", "-fPIC", "-Xptxas", "-v", "-I",
                        os.path.join(build.ROOT, "include")], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    m = re.search(r"Compiling entry function '\w*k_catchup\w*'.*?(\d+) bytes spill stores, (\d+) bytes spill loads",
                  r.stderr, re.S)
    assert m, r.stderr
    assert m.groups() == ("0", "0")
