"""FP32 x-lines of 256 points and more: 8 elements per thread up to 4096 lines, 16 above.

Fields of few lines are those of a plan with x_elems = 8 bit for bit, fields of more lines from 512 packed points on those
of x_elems = 16; 256 packed points take 16 in the forward pass only.
"""
import pytest
import torch

from paper_2010_14132_gb300 import workloads as wl
from paper_2010_14132_gb300.solver import Plan

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx", [512, 1024, 2048, 4096])
@pytest.mark.parametrize("ny,nz,chunk", [(8, 2, 0), (64, 8, 0), (256, 16, 0), (243, 17, 0), (256, 17, 0), (256, 17, 5)])
def test_elements_by_the_number_of_lines(nx, ny, nz, chunk):
    h = 8.0 / nx
    d = wl.random_stretched(nx, ny, nz, seed=nx + ny, dx=h, dy=h)
    S = torch.from_numpy(d.S).cuda().float()
    args = (nx, ny, nz, d.dx, d.dy, d.dz, d.rho0)
    p, e8, e16 = (Plan(*args, dtype="fp32", level_chunk=chunk, **o).solve(S)
                  for o in ({}, dict(x_elems=8), dict(x_elems=16)))
    assert not torch.equal(e8, e16)
    if ny * nz <= 4096:
        assert torch.equal(p, e8)
    elif nx >= 1024:
        assert torch.equal(p, e16)
    else:
        assert not torch.equal(p, e8) and not torch.equal(p, e16)
