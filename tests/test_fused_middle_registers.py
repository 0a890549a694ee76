"""Registers of the fused spectral middle (compiled here, no GPU): the CTAs per SM that its launch bounds ask for fit.

An SM has 65536 registers, handed out to a warp in units of 8 a thread.  CTAs of 128 threads at 256 points: three per SM,
168 registers a thread at most; 256 threads at 512 and 512 at 1024 points: two per SM, 128 and 64.
"""
import os
import re
import shutil
import subprocess

import pytest

from paper_2010_14132_gb300 import build as B


def test_ctas_per_sm(tmp_path):
    if not (shutil.which("nvcc") or os.path.exists("/usr/local/cuda/bin/nvcc")):
        pytest.skip("no nvcc")
    r = subprocess.run([B.nvcc(), *B._flags(["-Xptxas", "-v"]), "-c", os.path.join(B.CSRC, "spectral_fused.cu"), "-o",
                        str(tmp_path / "m.o")], capture_output=True, text=True, check=True)
    regs = re.findall(r"Compiling entry function '\w*k_midILi(\d+)E\w*'.*?Used (\d+) registers", r.stdout + r.stderr,
                      flags=re.S)
    assert len(regs) == 6
    for n, used in regs:
        n, used = int(n), (int(used) + 7) // 8 * 8
        threads, ctas = {256: (128, 3), 512: (256, 2), 1024: (512, 2)}[n]
        assert used * threads * ctas <= 65536, (n, used)
