"""FP64 solves of fields below the normal range of double: results are subnormal numbers, not zeros.

The solve is linear, so p(2^-s S) is 2^-s p(S) but for the roundings to multiples of u = 2^-1074.  With every stored
value off by at most u/2 a part, G the largest 1/|eigenvalue| and worst-case sums: the forward x-pass's values reach a
mode through ny terms and G, the y-pass's through G, a column's nz levels two roundings each straight into nx ny
terms, the inverse passes' nx terms and one.
"""
import numpy as np
import pytest
import torch

from paper_2010_14132_gb300 import workloads as wl
from paper_2010_14132_gb300.solver import Plan

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny", [(32, 32), (36, 24)])
@pytest.mark.parametrize("shift", [1030, 1040, 1046])
@pytest.mark.parametrize("x_kernel,y_kernel", [(0, 4), (1, 1)])   # fixed point, and the run-time FP64 engine
def test_scaled_solve(nx, ny, shift, x_kernel, y_kernel):
    nz = 8
    d = wl.Domain(nx, ny, nz, 1.0, 1.0, np.ones(nz), np.ones(nz), wl.normal_source((nz, ny, nx), seed=nx + ny))
    plan = Plan(nx, ny, nz, d.dx, d.dy, d.dz, d.rho0, dtype="fp64", x_kernel=x_kernel, y_kernel=y_kernel)
    # a source on the grid of 2^-24 around one: exact at every scale here
    S = torch.from_numpy(np.round(d.S * 2.0 ** 24) * 2.0 ** -24).cuda()
    u = 2.0 ** -1074
    G = 1.0 / (4 * np.sin(np.pi / max(nx, ny)) ** 2)
    bound = (G * (ny + 1) + nx * ny * 2 * (nz + 1) + nx + 1) * u * np.sqrt(0.5)
    small = S * 2.0 ** -500 * 2.0 ** (500 - shift)
    for f in (plan.solve, lambda x: plan.adjoint(x)[0]):
        p, q = f(S), f(small)
        # both in units of u: the scaled solution (exact: a power of two, up to the bound), and what came back
        want, got = p.cpu().numpy() * 2.0 ** (1074 - shift), q.cpu().numpy() * 2.0 ** 1000 * 2.0 ** 74
        assert np.abs(got).max() >= 2.0 ** (1074 - shift - 3)
        assert np.abs(got - want).max() <= bound / u + 2.0 ** -40 * np.abs(want).max()
