"""FP64 plans: the errors of the fixed-point transforms, against a solve in extended precision.

The reference is the same discrete problem in numpy's long double (library FFTs, one elimination per wavenumber column).
Every line length with fixed-point kernels is taken as x and as y line, with white noise, a dominant bin, an outlier, a
full-scale alternating field and a weak level; each level's error is taken relative to its own norm, and the largest, over
levels, of its rms over four seeds counts.

Limit, with u = 2^-53 and e the same error of the plan with FP64 butterflies: 8 u + 2 e.  Each of the four passes rounds
its results once, to at most u of each; the columns' eigenvalues, pivots and recurrences, the same code in both plans, give
some 4 u on columns as well conditioned as these (dx = 8/max(nx, ny)).  Where low wavenumbers amplify what the
transforms leave in them (up to max lambda / min lambda, 10^6 here, under the alternating field), the butterflies' 2^-53
sqrt(log2 n) of a line's norm stands against the fixed point's one rounding and 2^-62 sqrt(n), no more than that; what
is then compared are the errors of a handful of bins, whose rms over four seeds scatters by about a quarter: twice e.
"""
import numpy as np
import pytest
import torch

from paper_2010_14132_gb300 import workloads as wl
from paper_2010_14132_gb300.solver import Plan

pytestmark = pytest.mark.gpu

LENGTHS = [16, 18, 24, 32, 36, 48, 54, 64, 72, 96, 108, 128, 144, 192, 216, 256, 288, 324, 384, 432, 512, 576, 768, 864,
           1024, 2048]
SEEDS = 4
U = 2.0 ** -53


class Exact:
    """The discrete problem in long double."""

    def __init__(self, d):
        L = np.longdouble
        dz, rho, dx, dy = d.dz.astype(L), d.rho0.astype(L), L(d.dx), L(d.dy)
        self.nx, self.ny, self.nz = d.nx, d.ny, d.nz
        self.W, self.h, self.rf = rho * dz, (dz[1:] + dz[:-1]) / 2, (rho[1:] + rho[:-1]) / 2
        self.a = np.concatenate([[L(0)], self.rf / (self.W[1:] * self.h)])
        self.c = np.concatenate([self.rf / (self.W[:-1] * self.h), [L(0)]])
        pi, kx, ky = 4 * np.arctan(L(1)), np.arange(d.nx // 2 + 1).astype(L), np.arange(d.ny)
        ky = np.minimum(ky, d.ny - ky).astype(L)
        self.s = (4 / dy ** 2 * np.sin(pi * ky / d.ny) ** 2)[:, None] + (4 / dx ** 2 * np.sin(pi * kx / d.nx) ** 2)[None, :]

    def solve(self, S):
        F = np.fft.rfft2(S.astype(np.longdouble), axes=(1, 2))
        assert F.dtype == np.clongdouble
        f0 = F[:, 0, 0].real / (self.nx * self.ny)
        inv, g = np.empty_like(F.real), self.s.copy()
        for k in range(self.nz):
            if k:
                g = self.s + self.a[k] * (g * inv[k - 1])
                F[k] += self.a[k] * (F[k - 1] * inv[k - 1])
            u = g + self.c[k]
            u[0, 0] = 1   # solved apart below
            inv[k] = 1 / u
        F[-1] *= -inv[-1]
        for k in range(self.nz - 2, -1, -1):
            F[k] = (self.c[k] * F[k + 1] - F[k]) * inv[k]
        r = f0 - (self.W * f0).sum() / self.W.sum()   # the horizontal mean: fluxes summed upwards, then the pressure
        p0 = np.concatenate([[0], np.cumsum(np.cumsum(self.W * r)[:-1] * self.h / self.rf)])
        F[:, 0, 0] = (p0 - p0.mean()) * (self.nx * self.ny)
        return np.fft.irfft2(F, s=(self.ny, self.nx), axes=(1, 2))

    def adjoint(self, w):
        W = self.W[:, None, None]
        mu = W * self.solve((w - w.astype(np.longdouble).mean()) / W)
        return mu - W * (mu.sum() / (self.W.sum() * self.nx * self.ny))


def _sources(d, seed):
    rng = np.random.default_rng(seed)
    noise = rng.standard_normal((d.nz, d.ny, d.nx))
    i, j = np.arange(d.nx)[None, None, :], np.arange(d.ny)[None, :, None]
    outlier = noise.copy()
    outlier[d.nz // 2, d.ny // 3, d.nx // 5] = 1e10
    weak = noise.copy()
    weak[0] *= 1e-6
    return {"noise": noise, "bin": np.cos(2 * np.pi * i / d.nx) + 1e-3 * noise, "outlier": outlier,
            "alternating": (1.0 - 2.0 * ((i + j) % 2)) + 1e-3 * noise, "weak level": weak}


def _square(p, ref):
    e = p.cpu().numpy().astype(np.longdouble) - ref
    return ((e * e).sum((1, 2)) / (ref * ref).sum((1, 2))).astype(float)


@pytest.mark.parametrize("n", LENGTHS)
@pytest.mark.parametrize("axis", ["x", "y"])
def test_errors_against_extended_precision(n, axis):
    nx, ny, nz = (2 * n, 6, 3) if axis == "x" else (34 if n % 2 else 36, n, 3)
    h = 8.0 / max(nx, ny)
    d = wl.random_stretched(nx, ny, nz, seed=nx + 3 * ny, dx=h, dy=1.3 * h)
    ref = Exact(d)
    plans = [Plan(nx, ny, nz, d.dx, d.dy, d.dz, d.rho0, dtype="fp64", **o) for o in ({}, dict(x_kernel=1, y_kernel=1))]
    squares = {}
    for seed in range(SEEDS):
        for name, S in _sources(d, seed).items():
            St = torch.from_numpy(S).cuda()
            p, g = ref.solve(S), ref.adjoint(S)
            squares.setdefault((name, "solve"), []).append([_square(pl.solve(St), p) for pl in plans])
            squares.setdefault((name, "adjoint"), []).append([_square(pl.adjoint(St)[0], g) for pl in plans])
    for key, sq in squares.items():
        fixed, butterflies = np.sqrt(np.mean(sq, axis=0)).max(axis=1)   # [plan][level] -> [plan]
        assert fixed <= 8 * U + 2 * butterflies, (key, fixed / U, butterflies / U)
