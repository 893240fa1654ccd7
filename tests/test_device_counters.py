"""The counter of scanned arcs is written by kernels: it is handed down as a
device buffer, never as a bare pointer (a host variable's address would compile
as one, and only works where the GPU can reach host memory by itself)."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_1402_3281_gb300", "csrc")


def test_arc_counter_is_a_device_buffer():
    found = 0
    for f in ("common.cuh", "lp.cu", "driver.cu"):
        src = open(os.path.join(CSRC, f)).read()
        for m in re.finditer(r"void (?:lp_run|run_ip)\(([^)]*)\)", src):
            found += 1
            assert "DevBuf<int64_t>& arcs" in m.group(1), (f, m.group(0))
    assert found == 3
