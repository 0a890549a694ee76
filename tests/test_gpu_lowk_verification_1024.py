"""The low-wavenumber verification on grids of 1024-point y-lines, which mixed plans transform in two stages of radix 32.

As test_gpu_refinement.py has it for shorter lines: the first try's norm is at least the full verification's and at most 4
times it, both return the same iterate, and its bound holds, here against the FP64 plan.
"""
import numpy as np
import pytest
import torch

from paper_2010_14132_gb300 import workloads as wl
from paper_2010_14132_gb300.solver import Plan

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(512, 1024, 64), (1024, 1024, 64), (256, 1024, 48), (768, 1024, 40), (384, 1024, 33)])
@pytest.mark.parametrize("kind,seed", [("noise", 3), ("noise", 12), ("blobs", 11), ("blobs", 12)])
def test_low_wavenumber_bound(shape, kind, seed):
    d = (wl.anelastic_noise if kind == "noise" else wl.anelastic_blobs)(*shape, seed=seed)
    S = torch.from_numpy(np.ascontiguousarray(d.S)).cuda()
    (p, i), (q, j) = (Plan(*shape, d.dx, d.dy, d.dz, d.rho0, dtype="mixed", **kw).solve(S, info=True)
                      for kw in ({}, {"verify": 2}))
    ref = Plan(*shape, d.dx, d.dy, d.dz, d.rho0, dtype="fp64").solve(S)
    err = float((p - ref).norm() / ref.norm())
    assert i["converged"] and j["converged"] and err <= i["error_estimate"] <= 1e-10, (err, i, j)
    if i["sweeps"] == 1:
        assert torch.equal(p, q)
        assert i["rel_update"][2] >= j["rel_update"][2] * (1 - 1e-6), (i, j)
        assert i["rel_update"][2] <= 4 * j["rel_update"][2], (i, j)
    elif j["sweeps"] == 2:   # neither certified sweep 1's iterate
        assert torch.equal(p, q) and i["error_estimate"] == j["error_estimate"], (i, j)
