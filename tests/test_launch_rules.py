"""The launch rules of csrc/launch_rules.hpp, compiled by the host compiler (no GPU, no CUDA header)."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2010_14132_gb300", "csrc")


def _run(tmp_path, body):
    """Compile a main() around body, run it, return the lines it prints."""
    cxx = shutil.which("g++") or pytest.skip("no host C++ compiler")
    src, exe = tmp_path / "rules.cpp", tmp_path / "rules"
    src.write_text('#include <cstdio>\n#include <initializer_list>\n#include "launch_rules.hpp"\nusing namespace pgb;\nint main() {\n' + body + "}\n")
    subprocess.run([cxx, "-std=c++17", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    return subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.splitlines()


def test_warp_masks_name_existing_lanes_only(tmp_path):
    """Blocks of the column kernels (16 to 128 threads), and blocks whose last warp is partly filled."""
    lines = _run(tmp_path, """
  for (int n : {16, 20, 32, 48, 64, 100, 128})
    for (int t = 0; t < n; ++t) printf("%d %d %d %u\\n", n, t, warp_lanes(t, n), warp_mask(t, n));
""")
    assert len(lines) == 16 + 20 + 32 + 48 + 64 + 100 + 128
    for line in lines:
        n, t, lanes, mask = map(int, line.split())
        exists = [32 * (t // 32) + b < n for b in range(32)]
        assert lanes == sum(exists)
        assert mask == sum(1 << b for b in range(32) if exists[b]), line
