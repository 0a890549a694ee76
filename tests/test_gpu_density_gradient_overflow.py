"""Density gradient whose float products pass the float range: an infinity of the right sign, not NaN.

p is zero but at one point of the lowest level, so that only the face between levels 0 and 1 has terms:
dL/drho_0 = 0.5/(W_1 h) Up + 0.5 rho_1/rho_0 /(W_0 h) Lo and dL/drho_1 = -(0.5 rho_0/rho_1 /(W_1 h) Up + 0.5/(W_0 h) Lo),
h the face's height, with Lo = gS_0 (p_1 - p_0) and Up = gS_1 (p_1 - p_0) of one sign next to a point's adjoint field.
"""
import pytest
import torch

from paper_2010_14132_gb300 import workloads as wl
from paper_2010_14132_gb300.solver import Plan

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", ["fp32", "mixed"])
@pytest.mark.parametrize("sign", [1.0, -1.0])
def test_overflowing_products_give_infinities(dtype, sign):
    d = wl.random_stretched(32, 24, 6, seed=3)
    plan = Plan(d.nx, d.ny, d.nz, d.dx, d.dy, d.dz, d.rho0, dtype=dtype)
    gp = torch.zeros(plan.shape, dtype=plan.field_dtype, device="cuda")
    p = torch.zeros_like(gp)
    gp[0, 5, 7] = 1e15
    p[0, 5, 7] = sign * 1e30
    gS, grho = plan.adjoint(gp, p=p, want_grho=True)
    lo, up = (float(gS[k, 5, 7]) * -sign * 1e30 for k in (0, 1))
    assert lo * up > 0 and min(abs(lo), abs(up)) > 1e39
    inf = float("inf") if lo > 0 else -float("inf")
    assert float(grho[0]) == inf and float(grho[1]) == -inf, grho
    assert bool((grho[2:] == 0).all())
    # and within the range: the same formula, to the float products' rounding
    p[0, 5, 7] = sign
    gS, grho = plan.adjoint(gp, p=p, want_grho=True)
    lo, up = (float(gS[k, 5, 7]) * -sign for k in (0, 1))
    W, h = d.rho0 * d.dz, 0.5 * (d.dz[0] + d.dz[1])
    assert float(grho[0]) == pytest.approx(0.5 / (W[1] * h) * up + 0.5 * d.rho0[1] / d.rho0[0] / (W[0] * h) * lo, rel=1e-6)
    assert float(grho[1]) == pytest.approx(-(0.5 * d.rho0[0] / d.rho0[1] / (W[1] * h) * up + 0.5 / (W[0] * h) * lo), rel=1e-6)
