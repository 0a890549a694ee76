"""FP64 column solves: two half columns meeting in one warp against one thread per column.

The grids give one real part, one column or a pair of columns to a lane; the level counts are the smallest
ones, odd and even ones.  Both eliminations use subtraction-free pivots with errors of a few 2^-53 per entry on
columns as well conditioned as the parity tests' (dx = 8/max(nx, ny)): they agree to 1e-13 in the norm.
"""
import pytest
import torch

from paper_2010_14132_gb300 import workloads as wl
from paper_2010_14132_gb300.solver import Plan

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny", [(16, 12), (36, 27), (256, 96), (256, 256), (288, 243)])
@pytest.mark.parametrize("nz", [2, 3, 4, 5, 32, 65])
@pytest.mark.parametrize("bc", ["neumann", "dirichlet_top"])
def test_half_columns_agree_with_one_thread_per_column(nx, ny, nz, bc):
    h = 8.0 / max(nx, ny)
    d = wl.random_stretched(nx, ny, nz, seed=nx + ny + nz, dx=h, dy=1.3 * h)
    a, b = (Plan(nx, ny, nz, d.dx, d.dy, d.dz, d.rho0, dtype="fp64", bc=bc, col_tile=t) for t in (0, 16))
    S = torch.from_numpy(d.S).cuda()
    for f in (lambda pl: pl.solve(S), lambda pl: pl.adjoint(S)[0]):
        p, q = f(a), f(b)
        assert float((p - q).norm() / q.norm()) <= 1e-13
