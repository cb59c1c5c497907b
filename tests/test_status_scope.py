"""The kernels' status word lies in host memory, where the host may take and
clear it while a kernel of another stream still runs: every kernel writes it
through report(), in system scope.  Read off the sources, CPU only."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2601_16791_gb300", "csrc")


def test_status_word_is_written_in_system_scope():
    calls = 0
    for f in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        text = open(f).read()
        calls += len(re.findall(r"\breport\(", text))
        for m in re.finditer(r"\batomic\w+\(([^,;]*),", text):
            assert "status" not in m.group(1) or m.group(0).startswith("atomicOr_system("), (f, m.group(0))
    body = re.search(r"void report\(unsigned\* status, unsigned bits\) \{(.*?)\}",
                     open(os.path.join(CSRC, "mx_common.cuh")).read(), re.S)
    assert body and "atomicOr_system(status, bits)" in body.group(1)
    assert calls > 1
