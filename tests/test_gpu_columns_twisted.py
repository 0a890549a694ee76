"""Float column solves eliminated from both ends: the adjoint, and the double low-wavenumber columns.

The smallest level counts (one or no level above the meeting one), odd and even ones, both boundary conditions,
against the FP64 plan of the same grid; the mean column is among the low-wavenumber ones.  Tolerances: the parity
tests' (fp32 1e-5, mixed 1e-10), the mixed path's adjoint transforms floats.
"""
import pytest
import torch

from paper_2010_14132_gb300 import workloads as wl
from paper_2010_14132_gb300.solver import Plan

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny", [(12, 8), (64, 48)])
@pytest.mark.parametrize("nz", [2, 3, 4, 5, 33, 64, 129])
@pytest.mark.parametrize("bc", ["neumann", "dirichlet_top"])
def test_columns_from_both_ends(nx, ny, nz, bc):
    h = 8.0 / max(nx, ny)
    d = wl.random_stretched(nx, ny, nz, seed=nx + ny + nz, dx=h, dy=1.3 * h)
    args = (nx, ny, nz, d.dx, d.dy, d.dz, d.rho0)
    S = torch.from_numpy(d.S).cuda()
    ref = Plan(*args, dtype="fp64", bc=bc)
    p, g = ref.solve(S), ref.adjoint(S)[0]

    def off(a, b):
        return float((a.double() - b).norm() / b.norm())

    f = Plan(*args, dtype="fp32", bc=bc)
    assert off(f.solve(S.float()), p) <= 1e-5
    assert off(f.adjoint(S.float())[0], g) <= 1e-5
    m = Plan(*args, dtype="mixed", bc=bc)
    q, info = m.solve(S, info=True)
    assert info["converged"] and off(q, p) <= 1e-10
    assert off(m.adjoint(S)[0], g) <= 1e-5
