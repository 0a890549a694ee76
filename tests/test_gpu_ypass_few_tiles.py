"""FP32 y-lines of 512 points: 16 elements per thread with no more tiles (of 8 columns of a level) than SMs, 32 above.

Fields of few tiles are those of a plan with y_elems = 16 bit for bit; others are not, and with chunks of levels, column
counts that leave the last tile nearly empty and every tile width they are within the parity tests' 1e-5 of the FP64
solution.  1024 points take 32 with any number of tiles.
"""
import pytest
import torch

from paper_2010_14132_gb300 import workloads as wl
from paper_2010_14132_gb300.solver import Plan

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny,nz,opts", [
    (4, 512, 2, {}), (64, 512, 8, {}), (64, 512, 30, {}), (64, 512, 31, {}), (64, 512, 31, dict(level_chunk=7)),
    (64, 512, 30, dict(level_chunk=7)), (16, 512, 76, {}), (16, 512, 77, {}), (18, 512, 80, {}), (1024, 512, 2, {}),
    (1024, 512, 3, {}), (64, 512, 61, dict(y_tile=16)), (18, 512, 61, dict(y_tile=4)), (18, 512, 60, dict(y_tile=2)),
    (16, 1024, 2, {}), (64, 1024, 8, {})])
def test_elements_by_the_number_of_tiles(nx, ny, nz, opts):
    h = 8.0 / max(nx, ny)
    d = wl.random_stretched(nx, ny, nz, seed=nx + nz, dx=h, dy=h)
    S = torch.from_numpy(d.S).cuda()
    args = (nx, ny, nz, d.dx, d.dy, d.dz, d.rho0)
    p, e16 = (Plan(*args, dtype="fp32", **opts, **o).solve(S.float()) for o in ({}, dict(y_elems=16)))
    width = min(opts.get("y_tile", 8), 16 if ny == 512 else 8)
    tiles = -(-(nx // 2 + 1) // width) * nz
    few = ny == 512 and tiles <= torch.cuda.get_device_properties(0).multi_processor_count
    assert torch.equal(p, e16) == few
    ref = Plan(*args, dtype="fp64").solve(S)
    assert float((p.double() - ref).norm() / ref.norm()) <= 1e-5
