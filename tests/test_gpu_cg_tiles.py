"""Conjugate gradients on grids whose tiles are ragged, against the oracle's operator.

Tiles are 64 x 8 points and 16 levels: grids narrower than a tile, a last tile of a few points or of one row,
level counts around the tile's, both boundary conditions, and both preconditioner forms (float and double
fields).  A neighbour taken from the wrong place makes the operator unsymmetric or inconsistent with the oracle's,
so that the residual of the returned p, formed by the oracle in FP64, would stay far above the tolerance.
"""
import numpy as np
import pytest
import torch

import oracle as O
from paper_2010_14132_gb300 import workloads as wl
from paper_2010_14132_gb300.solver import Plan

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims", [(4, 4, 2), (6, 9, 3), (64, 8, 16), (96, 27, 17), (162, 9, 33), (128, 81, 5),
                                  (4, 81, 4), (192, 12, 15)])
@pytest.mark.parametrize("bc", ["neumann", "dirichlet_top"])
@pytest.mark.parametrize("dtype,opts", [("fp64", {}), ("mixed", {"max_sweeps": 0}), ("mixed", {})])
def test_ragged_tiles(dims, bc, dtype, opts):
    d = wl.random_stretched(*dims, seed=sum(dims))
    rho3 = wl.perturbed_density(d.nx, d.ny, d.rho0, 0.2, seed=9)
    plan = Plan(*dims, d.dx, d.dy, d.dz, rho3.mean(axis=(1, 2)), dtype=dtype, bc=bc, **opts)
    p, info = plan.cg_solve(torch.from_numpy(rho3).cuda(), torch.from_numpy(d.S).cuda(), tol=1e-10, max_iter=100)
    assert info["converged"], info
    S = d.S
    if bc == "neumann":
        W = O.weights_var(d.dz, rho3)
        S = S - (W * S).sum() / W.sum()
    r = S - O.apply_A_var(p.cpu().numpy(), d.dx, d.dy, d.dz, rho3, bc)
    # the recursive residual's distance from the true one stays below the tolerance itself
    assert np.linalg.norm(r) / np.linalg.norm(d.S) <= 2e-10
