"""FP32 x-lines of 256 points and more: 16 elements per thread by default, against the choices that can be set.

Row counts that leave the last group of rows short (a group is 8 rows of 256 points, 4 of 512, 2 of 1024, one of
2048), against the FP64 plan.  Every FP32 form is within the parity tests' 1e-5 of the exact solution, and so within
2e-5 of the others; a form that is set explicitly is bitwise the same on every call.
"""
import pytest
import torch

from paper_2010_14132_gb300 import workloads as wl
from paper_2010_14132_gb300.solver import Plan

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx", [256, 512, 1024, 2048, 4096])
@pytest.mark.parametrize("ny,nz", [(6, 3), (9, 5)])
def test_default_elements(nx, ny, nz):
    h = 8.0 / nx
    d = wl.random_stretched(nx, ny, nz, seed=nx + ny, dx=h, dy=h)
    S = torch.from_numpy(d.S).cuda()
    args = (nx, ny, nz, d.dx, d.dy, d.dz, d.rho0)
    ref = Plan(*args, dtype="fp64").solve(S)
    p = Plan(*args, dtype="fp32").solve(S.float()).double()
    assert float((p - ref).norm() / ref.norm()) <= 1e-5
    for e in (8, 16):
        plan = Plan(*args, dtype="fp32", x_elems=e)
        q = plan.solve(S.float())
        assert torch.equal(q, plan.solve(S.float()))
        assert float((p - q.double()).norm() / ref.norm()) <= 2e-5
