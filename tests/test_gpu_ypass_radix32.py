"""FP32 y-lines of 512 and 1024 points: the two-stage form with 32 elements per thread.

Column counts that leave the last tile nearly empty (9, 10 and 33 columns), every tile width, both directions (a
solve runs each once), against the form with 8 elements per thread and the FP64 plan.  Both FP32 forms are within
the parity tests' 1e-5 of the exact solution, and so within 2e-5 of each other.
"""
import pytest
import torch

from paper_2010_14132_gb300 import workloads as wl
from paper_2010_14132_gb300.solver import Plan

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ny", [512, 1024])
@pytest.mark.parametrize("nx", [16, 18, 64])
@pytest.mark.parametrize("tile", [None, 2, 4, 8, 16])
def test_two_stage_ypass(nx, ny, tile):
    nz = 3
    h = 8.0 / ny
    d = wl.random_stretched(nx, ny, nz, seed=ny + nx, dx=h, dy=h)
    S = torch.from_numpy(d.S).cuda()
    args = (nx, ny, nz, d.dx, d.dy, d.dz, d.rho0)
    ref = Plan(*args, dtype="fp64").solve(S)
    p = Plan(*args, dtype="fp32", y_tile=tile).solve(S.float()).double()
    assert float((p - ref).norm() / ref.norm()) <= 1e-5
    q = Plan(*args, dtype="fp32", y_elems=8).solve(S.float()).double()
    assert float((p - q).norm() / ref.norm()) <= 2e-5
