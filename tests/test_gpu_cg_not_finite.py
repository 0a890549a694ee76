"""Conjugate gradients on input that is not finite: not converged, and p is the iterate before the failed step.

With a NaN in the source or the density the first direction has no step (d . K d is NaN), so p is the initial guess,
zero everywhere; with a negative density d . K d is negative and it ends the same way.
"""
import numpy as np
import pytest
import torch

from paper_2010_14132_gb300 import workloads as wl
from paper_2010_14132_gb300.solver import Plan

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("where", ["source", "density", "sign"])
@pytest.mark.parametrize("bc", ["neumann", "dirichlet_top"])
@pytest.mark.parametrize("dtype,opts", [("fp64", {}), ("mixed", {"max_sweeps": 0}), ("mixed", {})])
def test_p_stays_at_the_last_iterate(where, bc, dtype, opts):
    d = wl.random_stretched(24, 16, 6, seed=5)
    rho3 = wl.perturbed_density(d.nx, d.ny, d.rho0, 0.1, seed=6)
    plan = Plan(d.nx, d.ny, d.nz, d.dx, d.dy, d.dz, d.rho0, dtype=dtype, bc=bc, **opts)
    S = d.S.copy()
    if where == "source":
        S[3, 5, 7] = np.nan
    elif where == "density":
        rho3[2, 4, 9] = np.nan
    else:
        rho3 = -rho3
    p, info = plan.cg_solve(torch.from_numpy(rho3).cuda(), torch.from_numpy(S).cuda(),
                            out=torch.full(d.S.shape, 7.0, dtype=torch.float64, device="cuda"))
    assert not info["converged"], info
    assert bool((p == 0).all())
