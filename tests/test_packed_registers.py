"""The request server's packed kernel inlines the bodies of every law into 64 registers a
thread, so a body that grows makes all of them spill. The bounds are those of the build
whose 128^3 LPS request alone took 0.573 ms a step; with 496 bytes of spill stores it
took 0.617."""
import os
import re
import subprocess

import pytest

from paper_1806_06917_gb300 import build as B


def test_packed_kernel_spills_no_more_than_measured(tmp_path):
    nvcc = B.nvcc()
    try:
        subprocess.run([nvcc, "--version"], capture_output=True, check=True)
    except (OSError, subprocess.CalledProcessError):
        pytest.skip("no nvcc")
    cmd = [nvcc] + B.ARCH + B.FLAGS + ["-Xptxas", "-v", "-c", os.path.join(B.CSRC, "pd_packed.cu"), "-o",
                                       str(tmp_path / "pd_packed.o")]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    m = re.search(r"pd_packed_round.*?(\d+) bytes stack frame, (\d+) bytes spill stores, (\d+) bytes spill loads",
                  r.stdout + r.stderr, re.S)
    assert m, "no resource report of pd_packed_round"
    _, stores, loads = map(int, m.groups())
    assert stores <= 196 and loads <= 528, "pd_packed_round spills %d bytes of stores, %d of loads" % (stores, loads)
