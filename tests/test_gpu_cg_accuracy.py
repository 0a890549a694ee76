"""The accuracy that conjugate gradients reach when they are not stopped: the error of the operator's double-float form.

Iterated to a tolerance below that error, the recursive residual goes on falling while the true one, formed by the
oracle in FP64 (whose own rounding is a hundred times smaller), stays where the operator's errors have left it: it
repeats to a few per cent.  The limits are the values that the operator gave with its face coefficients formed in
FP64 (one rounding of the sum, then split into float pairs): the form that sums densities already split has to be no
further off.
"""
import numpy as np
import pytest
import torch

import oracle as O
from paper_2010_14132_gb300 import workloads as wl
from paper_2010_14132_gb300.solver import Plan

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims,bc,seed,limit", [((64, 64, 32), "neumann", 1, 7.26e-14),
                                                ((96, 32, 24), "neumann", 1, 1.16e-13),
                                                ((64, 48, 101), "dirichlet_top", 1, 2.78e-13),
                                                ((128, 128, 16), "neumann", 3, 2.42e-13)])
def test_attainable_residual(dims, bc, seed, limit):
    d = wl.anelastic_noise(*dims, seed=seed)
    rho3 = wl.perturbed_density(d.nx, d.ny, d.rho0, 0.2, seed=seed)
    plan = Plan(*dims, d.dx, d.dy, d.dz, rho3.mean(axis=(1, 2)), dtype="fp64", bc=bc)
    p, info = plan.cg_solve(torch.from_numpy(rho3).cuda(), torch.from_numpy(d.S).cuda(), tol=1e-15, max_iter=40)
    assert info["converged"], info
    S = d.S
    if bc == "neumann":
        W = O.weights_var(d.dz, rho3)
        S = S - (W * S).sum() / W.sum()
    r = S - O.apply_A_var(p.cpu().numpy(), d.dx, d.dy, d.dz, rho3, bc)
    assert np.linalg.norm(r) / np.linalg.norm(d.S) <= limit
