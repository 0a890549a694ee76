"""FP32 and mixed solves on short line lengths and ones with factors 9, 27 and 81 (compile-time transforms).

Each length is taken as the x line (nx = 2 N, lines that do not tile warps among them) and as the y line, with
row counts that leave the last group of rows short, against the FP64 plan of the same grid.  The tolerances
are the parity tests' (fp32 1e-5, mixed 1e-10), on columns as well conditioned as theirs (dx = 8/max(nx, ny)).
"""
import pytest
import torch

from paper_2010_14132_gb300 import workloads as wl
from paper_2010_14132_gb300.solver import Plan

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("axis,n", [("x", n) for n in (16, 18, 24, 36, 48, 54, 72, 108, 144, 216, 288, 324, 432)]
                         + [("y", n) for n in (32, 36, 48, 54, 72, 108, 144, 216, 288, 324, 432, 576, 864)])
@pytest.mark.parametrize("iso", [True, False])
def test_ragged_lengths(axis, n, iso):
    nx, ny, nz = (2 * n, 18, 5) if axis == "x" else (48, n, 5)
    h = 8.0 / max(nx, ny)
    d = wl.random_stretched(nx, ny, nz, seed=n, dx=h, dy=h if iso else 1.3 * h)
    S = torch.from_numpy(d.S).cuda()
    args = (nx, ny, nz, d.dx, d.dy, d.dz, d.rho0)
    ref = Plan(*args, dtype="fp64").solve(S)
    p = Plan(*args, dtype="fp32").solve(S.float())
    assert float((p.double() - ref).norm() / ref.norm()) <= 1e-5
    p, info = Plan(*args, dtype="mixed").solve(S, info=True)
    assert info["converged"]
    assert float((p - ref).norm() / ref.norm()) <= 1e-10
    plain = Plan(*args, dtype="mixed", x_kernel=1, y_kernel=1).solve(S)   # run-time line lengths
    assert float((p - plain).norm() / ref.norm()) <= 2e-10
