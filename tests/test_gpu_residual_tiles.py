"""Mixed solves whose residual passes stage every stencil row: row groups at the edges of a level.

Two to 32 rows a group (nx from 1536 down to 64), levels with fewer rows than a group, a short last group,
groups that touch both ends of the periodic direction, one level above or below only, level chunks.  A row
taken from the wrong place leaves a residual of the order of the source, and the refinement then ends above the
tolerance that is checked against the FP64 plan (1e-10, the mixed path's).
"""
import pytest
import torch

from paper_2010_14132_gb300 import workloads as wl
from paper_2010_14132_gb300.solver import Plan

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny,nz", [(32, 48, 3), (36, 16, 2), (48, 81, 2), (108, 32, 2), (64, 4, 2), (64, 36, 3), (64, 54, 2), (128, 48, 5), (192, 18, 2), (256, 27, 3),
                                      (432, 16, 4), (512, 6, 2), (1024, 4, 2), (1024, 9, 3), (1024, 128, 2),
                                      (1536, 9, 3), (2048, 8, 3)])
@pytest.mark.parametrize("opts", [{}, {"bc": "dirichlet_top"}, {"verify": 0}, {"level_chunk": 2}])
@pytest.mark.parametrize("iso", [True, False])
def test_row_groups(nx, ny, nz, opts, iso):
    h = 8.0 / max(nx, ny)
    d = wl.random_stretched(nx, ny, nz, seed=nx + ny + nz, dx=h, dy=h if iso else 1.3 * h)
    args = (nx, ny, nz, d.dx, d.dy, d.dz, d.rho0)
    S = torch.from_numpy(d.S).cuda()
    ref = Plan(*args, dtype="fp64", bc=opts.get("bc", "neumann")).solve(S)
    p, info = Plan(*args, dtype="mixed", **opts).solve(S, info=True)
    assert info["converged"], info
    err = float((p - ref).norm() / ref.norm())
    assert err <= 1e-10 and err <= info["error_estimate"], (err, info)
