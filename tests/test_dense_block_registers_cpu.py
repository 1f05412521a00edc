"""The dense-block kernels keep their tiles in registers: none of them spills."""
import os
import re
import subprocess

from paper_1412_2293_gb300 import build


def test_no_spills(tmp_path):
    r = subprocess.run([build._nvcc(), *build.ARCH, *build.FLAGS, "-Xptxas", "-v", "-c", os.path.join(build.CSRC, "tc.cu"),
                        "-o", str(tmp_path / "tc.o")], capture_output=True, text=True, check=True)
    spills = re.findall(r"k_dense_tc.*\n.*?(\d+) bytes spill stores, (\d+) bytes spill loads", r.stderr)
    assert len(spills) == 9, r.stderr[-2000:]                       # k = 3..5, three modes
    assert all(s == ("0", "0") for s in spills), spills
