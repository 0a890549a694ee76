"""Low-wavenumber columns solved by a block of half a warp (column kernels of 16 columns per CTA).

Their sums and the meeting of the two halves name the block's existing lanes only.  col_tile 16 is half a warp in every
type; col_tile 3 falls to it above 102 levels.  The removed mean and the solution against the default kernels': the
same right-hand side to the rounding of a tree of another shape (nz additions of a level sum: within 1e-13), the
solutions at the other column tests' tolerances.
"""
import pytest
import torch

from paper_2010_14132_gb300 import workloads as wl
from paper_2010_14132_gb300.solver import Plan

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype,tol", [("fp64", 1e-13), ("fp32", 1e-5), ("mixed", 2e-10)])
@pytest.mark.parametrize("col_tile,nz", [(16, 2), (16, 15), (16, 16), (16, 33), (3, 103), (16, 103)])
@pytest.mark.parametrize("bc", ["neumann", "dirichlet_top"])
def test_half_warp_blocks_agree_with_the_default(dtype, tol, col_tile, nz, bc):
    nx, ny = 48, 32
    d = wl.random_stretched(nx, ny, nz, seed=nz, dx=0.25, dy=0.3)
    a, b = (Plan(nx, ny, nz, d.dx, d.dy, d.dz, d.rho0, dtype=dtype, bc=bc, col_tile=t) for t in (col_tile, 0))
    # a mean of the size of the level means (1/sqrt(nx ny)): the solution carries the removed mean's rounding times the
    # square of the depth, here 125^2/2 x 2^-6 x 2^-53 = 1e-14
    S = (torch.from_numpy(d.S) + 2.0 ** -6).cuda().to(a.field_dtype)
    (p, ip), (q, iq) = (pl.solve(S, info=True) for pl in (a, b))
    assert float((p.double() - q.double()).norm() / q.double().norm()) <= tol
    if bc == "neumann":
        assert ip["removed_weighted_mean"] == pytest.approx(iq["removed_weighted_mean"], rel=1e-13)
        assert abs(float(p.double().mean())) <= tol * float(q.double().abs().max())
    g, h = a.adjoint(S)[0].double(), b.adjoint(S)[0].double()
    assert float((g - h).norm() / h.norm()) <= max(tol, 1e-5 if dtype == "mixed" else 0)
