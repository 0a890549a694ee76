"""FP64 plans: the fixed-point transforms against the FP64 butterflies and against exact scaling.

Every line length that has fixed-point kernels is taken once as the x line (nx = 2 N) and once as the y line;
sources are white noise, a spike, a single wave, rows of zeros among others, and lines of widely spread
magnitudes.  Both paths transform with errors of a few 2^-53 of a line's norm, on columns as well conditioned
as the parity tests' (dx = 8/max(nx, ny)), so they agree to 1e-14 in the norm.  The scale of a line is a power
of two, so scaling the source by a power of two scales the solution bit for bit.
"""
import numpy as np
import pytest
import torch

from paper_2010_14132_gb300 import workloads as wl
from paper_2010_14132_gb300.solver import Plan

pytestmark = pytest.mark.gpu

LENGTHS = [16, 18, 24, 32, 36, 48, 54, 64, 72, 96, 108, 128, 144, 192, 216, 256, 288, 324, 384, 432, 512, 576, 768, 864,
           1024, 2048]


def _domain(nx, ny, nz):
    h = 8.0 / max(nx, ny)
    return wl.random_stretched(nx, ny, nz, seed=nx + 3 * ny + nz, dx=h, dy=1.3 * h)


def _plan(d, **opts):
    return Plan(d.nx, d.ny, d.nz, d.dx, d.dy, d.dz, d.rho0, dtype="fp64", **opts)


def _sources(d):
    rng = np.random.default_rng(d.nx * 5 + d.ny)
    shape = (d.nz, d.ny, d.nx)
    spike = np.zeros(shape)
    spike[d.nz // 2, d.ny // 3, d.nx // 5] = -3.0
    wave = np.cos(2 * np.pi * np.arange(d.nx) / d.nx)[None, None, :] * np.ones(shape)
    rows = rng.standard_normal(shape)
    rows[:, ::2] = 0.0
    spread = np.exp(rng.normal(0, 6, shape))
    return {"noise": d.S, "spike": spike, "wave": wave, "rows": rows, "spread": spread}


@pytest.mark.parametrize("n", LENGTHS)
@pytest.mark.parametrize("axis", ["x", "y"])
def test_fixed_point_transforms_agree_with_fp64_butterflies(n, axis):
    d = _domain(2 * n, 6, 3) if axis == "x" else _domain(34 if n % 2 else 36, n, 3)
    a, b = _plan(d), _plan(d, x_kernel=1, y_kernel=1)
    for name, S in _sources(d).items():
        St = torch.from_numpy(S).cuda()
        p, q = a.solve(St), b.solve(St)
        assert float((p - q).norm() / q.norm()) <= 1e-14, name
        gp, gq = a.adjoint(St)[0], b.adjoint(St)[0]
        assert float((gp - gq).norm() / gq.norm()) <= 1e-14, name


@pytest.mark.parametrize("k", [-960, -900, -300, 1, 300, 900])
def test_power_of_two_scaling_is_exact(k):
    d = _domain(64, 48, 5)
    plan = _plan(d)
    S = torch.from_numpy(d.S).cuda()
    assert torch.equal(plan.solve(S * 2.0 ** k), plan.solve(S) * 2.0 ** k)


@pytest.mark.parametrize("value", [float("nan"), float("inf"), -float("inf")])
def test_non_finite_values_reach_the_whole_field(value):
    d = _domain(64, 48, 5)
    S = torch.from_numpy(d.S.copy()).cuda()
    S[2, 11, 17] = value
    assert not bool(torch.isfinite(_plan(d).solve(S)).any())
    assert not bool(torch.isfinite(_plan(d, x_kernel=1, y_kernel=1).solve(S)).any())


def test_zero_source_gives_zero():
    d = _domain(64, 48, 5)
    p = _plan(d).solve(torch.zeros((5, 48, 64), dtype=torch.float64, device="cuda"))
    assert not bool(p.any())


def test_level_chunks_give_the_same_bits():
    d = _domain(96, 64, 11)
    S = torch.from_numpy(d.S).cuda()
    assert torch.equal(_plan(d).solve(S), _plan(d, level_chunk=3).solve(S))
