"""Workspaces of grids that just fit the fixed array of poisson_solve_static_workspace (32 MiB).

The refinement's sums belong to mixed plans alone and hold a launch's blocks, not a slot for every group of rows, so that
these grids (each type, with and without low-wavenumber columns) keep within the array; and with level chunks the blocks
of all chunks share those slots.
"""
import numpy as np
import pytest
import torch

from paper_2010_14132_gb300 import _native as N
from paper_2010_14132_gb300 import workloads as wl
from paper_2010_14132_gb300.solver import Plan

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny,nz,dtype,opts", [
    (648, 576, 11, "fp64", {}), (864, 384, 24, "fp32", {}), (32, 1458, 89, "fp32", {}), (576, 1944, 7, "fp32", {}),
    (432, 768, 24, "fp32", {}), (36, 486, 125, "mixed", {}), (48, 288, 181, "mixed", dict(lowk_radius2=0)),
    (576, 16, 296, "mixed", dict(lowk_radius2=0)), (576, 128, 37, "mixed", dict(lowk_radius2=0))])
def test_grids_that_fit_the_static_workspace(nx, ny, nz, dtype, opts):
    d = wl.random_stretched(nx, ny, nz, seed=nz, dx=0.3, dy=0.3)
    plan = Plan(nx, ny, nz, d.dx, d.dy, d.dz, d.rho0, dtype=dtype, **opts)
    assert plan.workspace_bytes() <= N.POISSON_STATIC_WORKSPACE_BYTES
    S = torch.from_numpy(d.S).cuda().to(plan.field_dtype)
    p = torch.empty_like(S)
    st = N.poisson_solve_static_workspace(plan._h, S.data_ptr(), p.data_ptr(), torch.cuda.current_stream().cuda_stream)
    assert st in (N.POISSON_OK, N.POISSON_ERR_NOT_CONVERGED)
    q = plan.solve(S)
    assert torch.equal(p, q)


@pytest.mark.parametrize("nx,ny,nz", [(64, 64, 48), (256, 48, 37), (432, 24, 20)])
@pytest.mark.parametrize("chunk", [1, 5, 19])
def test_residual_sums_of_level_chunks(nx, ny, nz, chunk):
    """Chunked launches share the slots: the reported residuals, their sums, are those of one launch."""
    d = wl.anelastic_noise(nx, ny, nz, seed=nz)
    a, b = (Plan(nx, ny, nz, d.dx, d.dy, d.dz, d.rho0, dtype="mixed", max_sweeps=3, tolerance=1e-300, level_chunk=c)
            for c in (chunk, 0))
    S = torch.from_numpy(np.ascontiguousarray(d.S)).cuda()
    ip, iq = a.solve(S, info=True)[1], b.solve(S, info=True)[1]
    # float sums of nx/2 to 24000 squares a block, in another grouping
    assert ip["rel_residual"][:3] == pytest.approx(iq["rel_residual"][:3], rel=1e-4)
