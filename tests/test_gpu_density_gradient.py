"""The rho0 gradient's reductions against their defining sums in FP64 torch.

dL/drho0_m is a combination of Lo_f = sum g_k (p_{k+1} - p_k) and Up_f = sum g_{k+1} (p_{k+1} - p_k) over the
faces next to level m, g = dL/dS.  The sizes cover the splits of a level plane over blocks: less than one
block, whole blocks with a remainder, several points per thread.  Each term is rounded a few times, to double
or (float plans) to float, so the error is at most a few units of that precision times the sum of the
terms' magnitudes; the sums themselves run in double or in pairs of floats.
"""
import numpy as np
import pytest
import torch

from paper_2010_14132_gb300 import workloads as wl
from paper_2010_14132_gb300.solver import Plan

pytestmark = pytest.mark.gpu


def _reference(g, p, dz, rho):
    """(gradient, sum of the magnitudes of its terms), FP64."""
    t = lambda v: torch.from_numpy(np.asarray(v)).cuda()  # noqa: E731
    W, h, rf = t(rho * dz), t(0.5 * (dz[1:] + dz[:-1])), t(0.5 * (rho[1:] + rho[:-1]))
    D = p[1:] - p[:-1]
    lo, up = g[:-1] * D, g[1:] * D
    a, c = rf / (W[1:] * h), rf / (W[:-1] * h)   # a_{f+1}, c_f of face f
    up_above, up_below, lo_below, lo_above = (0.5 / (W[1:] * h) - a / t(rho)[1:], 0.5 / (W[1:] * h),
                                              0.5 / (W[:-1] * h) - c / t(rho)[:-1], 0.5 / (W[:-1] * h))
    grad, size = (torch.zeros(len(dz), dtype=torch.float64, device="cuda") for _ in range(2))
    lo_s, up_s, lo_m, up_m = (v.sum(dim=(1, 2)) for v in (lo, up, lo.abs(), up.abs()))
    grad[1:] += up_above * up_s - lo_above * lo_s
    grad[:-1] += up_below * up_s - lo_below * lo_s
    # the two parts of a coefficient are rounded before they are subtracted
    size[1:] += (0.5 / (W[1:] * h) + a / t(rho)[1:]) * up_m + lo_above * lo_m
    size[:-1] += up_below * up_m + (0.5 / (W[:-1] * h) + c / t(rho)[:-1]) * lo_m
    return grad, size


@pytest.mark.parametrize("dims", [(4, 4, 2), (6, 4, 3), (18, 27, 40), (64, 48, 16), (128, 96, 5), (512, 512, 3)])
@pytest.mark.parametrize("dtype,unit", [("fp64", 2.0 ** -50), ("fp32", 2.0 ** -21), ("mixed", 2.0 ** -21)])
def test_density_gradient_sums(dims, dtype, unit):
    nx, ny, nz = dims
    d = wl.random_stretched(nx, ny, nz, seed=sum(dims))
    plan = Plan(nx, ny, nz, d.dx, d.dy, d.dz, d.rho0, dtype=dtype)
    gen = torch.Generator(device="cuda").manual_seed(5)
    w, p = (torch.randn((nz, ny, nx), generator=gen, device="cuda", dtype=torch.float64).to(plan.field_dtype)
            for _ in range(2))
    gS, grho = plan.adjoint(w, p=p, want_grho=True)
    ref, size = _reference(gS.double(), p.double(), d.dz, d.rho0)
    assert bool(((grho - ref).abs() <= unit * size).all()), ((grho - ref).abs() / size).max()
