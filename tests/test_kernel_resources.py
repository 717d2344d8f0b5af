"""What the compiler says of the operator kernels (-Xptxas -v): the float64 passes spill nothing.

They are compiled for six or eight resident blocks an SM, which leaves 40 or fewer registers a
thread; a spilled register costs memory traffic in the loops that bound a solve.
"""
import os
import re
import shutil
import subprocess

import pytest

from paper_2405_03584_gb300 import build


@pytest.mark.skipif(shutil.which("nvcc") is None, reason="no nvcc")
def test_operator_passes_do_not_spill(tmp_path):
    r = subprocess.run([shutil.which("nvcc"), *build.ARCH, *build.FLAGS, "-Xptxas", "-v", "-c",
                        os.path.join(build.CSRC, "kernels.cu"), "-o", str(tmp_path / "k.o")], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-2000:]
    found = re.findall(r"Compiling entry function '(\S+)'.*?\n.*?\n\s+\d+ bytes stack frame, (\d+) bytes spill stores, "
                       r"(\d+) bytes spill loads", r.stderr)
    passes = [f for f in found if re.search(r"k_op_(cols|rows)", f[0])]
    assert len(passes) >= 24 + 8, len(passes)
    assert [f for f in passes if f[1:] != ("0", "0")] == []
