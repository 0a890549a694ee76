"""The pressure-solve workloads whose speed matters, as a program calls them.

Each listed case is one call (or one training step) through the public torch API on a grid of the kind
the library is used on: periodic horizontal sizes 2^a 3^b, stretched or uniform vertical levels, an
anelastic density profile. `draw` gives further cases of the same ranges. `exact` states the same
problems in plain torch at 64 bits (library FFTs, one elimination per wavenumber column).
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2010_14132_gb300.solver import Batch, Plan, poisson_solve
from paper_2010_14132_gb300.workloads import Domain


def listed():
    return [
        # a small uniform box in double, solved once per timestep of a test or a teaching model: latency
        dict(name="solve_fp64_32x32x32", kind="solve", nx=32, ny=32, nz=32, dtype="fp64", dx=1.0, dy=1.0,
             levels="uniform", bc="neumann", layout="zyx", source="noise"),
        # the local domain of one large-eddy column model, mixed precision: latency
        dict(name="solve_mixed_64x64x48", kind="solve", nx=64, ny=64, nz=48, dtype="mixed", dx=50.0, dy=50.0,
             levels="stretched", bc="neumann", layout="zyx", source="blobs"),
        # an ordinary boundary-layer grid, single and double precision
        dict(name="solve_fp32_256x256x64", kind="solve", nx=256, ny=256, nz=64, dtype="fp32", dx=50.0, dy=50.0,
             levels="stretched", bc="neumann", layout="zyx", source="blobs"),
        dict(name="solve_fp64_256x256x64", kind="solve", nx=256, ny=256, nz=64, dtype="fp64", dx=50.0, dy=50.0,
             levels="stretched", bc="neumann", layout="zyx", source="blobs"),
        # a ragged grid (line lengths 216 and 324, an odd level count, dx != dy) in single precision
        dict(name="solve_fp32_432x324x37", kind="solve", nx=432, ny=324, nz=37, dtype="fp32", dx=40.0, dy=60.0,
             levels="stretched", bc="neumann", layout="zyx", source="noise"),
        # a host model that keeps its fields z-fastest and has p = 0 at its lid; odd level count, 3-smooth sizes
        dict(name="solve_mixed_384x192x75_zfast_lid", kind="solve", nx=384, ny=192, nz=75, dtype="mixed", dx=50.0,
             dy=75.0, levels="stretched", bc="dirichlet_top", layout="xyz", source="noise"),
        # training a closure through the projection: forward and backward, double with the density gradient too
        dict(name="grad_fp64_512x512x64", kind="grad", nx=512, ny=512, nz=64, dtype="fp64", dx=50.0, dy=50.0,
             levels="stretched", source="blobs", density=True),
        # the same in single precision, differentiated in the source alone
        dict(name="grad_fp32_512x512x64", kind="grad", nx=512, ny=512, nz=64, dtype="fp32", dx=50.0, dy=50.0,
             levels="stretched", source="blobs", density=False),
        # an ensemble of unequal domains advanced together
        dict(name="batch_mixed_24_uneven", kind="batch", domains=24, shapes=7, dtype="mixed"),
        # density that also varies in x and y: conjugate gradients around the direct solve
        dict(name="cg_mixed_512x512x64", kind="cg", nx=512, ny=512, nz=64, dx=50.0, dy=50.0, levels="stretched",
             perturbation=0.1),
        # the large grid: single precision, and mixed precision certified to 1e-10
        dict(name="solve_fp32_1024x1024x128", kind="solve", nx=1024, ny=1024, nz=128, dtype="fp32", dx=50.0,
             dy=50.0, levels="stretched", bc="neumann", layout="zyx", source="noise"),
        dict(name="solve_mixed_1024x1024x128", kind="solve", nx=1024, ny=1024, nz=128, dtype="mixed", dx=50.0,
             dy=50.0, levels="stretched", bc="neumann", layout="zyx", source="noise"),
    ]


# horizontal sizes of the form 2^a 3^b that models use
SIZES = sorted(2 ** a * 3 ** b for a in range(1, 11) for b in range(0, 4) if 32 <= 2 ** a * 3 ** b <= 1024)
MOST_POINTS = {"fp32": 1024 * 1024 * 128, "mixed": 1024 * 1024 * 128, "fp64": 512 * 512 * 96}


def _log_size(rng, lo=32, hi=1024):
    t = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    return min(SIZES, key=lambda n: abs(math.log(n / t)))


def draw(rng):
    kind = rng.choice(["solve", "solve", "solve", "solve", "grad", "grad", "batch", "cg"])
    if kind == "batch":
        return dict(kind="batch", domains=rng.randint(4, 24), shapes=rng.randint(100, 10 ** 6),
                    dtype=rng.choice(["mixed", "mixed", "fp32"]))
    dtype = "mixed" if kind == "cg" else rng.choice(["fp64", "fp32"] if kind == "grad" else ["fp64", "fp32", "mixed"])
    most = 512 * 512 * 64 if kind in ("cg", "grad") else MOST_POINTS[dtype]
    while True:
        nx = _log_size(rng)
        ny = nx if rng.random() < 0.4 else _log_size(rng)
        nz = rng.choice([16, 24, 31, 32, 48, 57, 64, 75, 96, 101, 128])
        if nx * ny * nz <= most and nx <= 8 * ny and ny <= 8 * nx:
            break
    dx = float(rng.choice([25, 50, 100]))
    case = dict(kind=kind, nx=nx, ny=ny, nz=nz, dx=dx, dy=dx if rng.random() < 0.6 else 1.5 * dx,
                levels=rng.choice(["stretched", "stretched", "uniform"]))
    if kind == "cg":
        return dict(case, perturbation=round(rng.uniform(0.02, 0.2), 3))
    case.update(dtype=dtype, source=rng.choice(["noise", "blobs"]))
    if kind == "grad":
        return dict(case, density=dtype == "fp64" and rng.random() < 0.5)
    return dict(case, bc="dirichlet_top" if rng.random() < 0.25 else "neumann",
                layout="xyz" if rng.random() < 0.25 else "zyx")


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

def _levels(case):
    """Thicknesses and densities: dz = 10 * 1.03^k m (uniform: the horizontal spacing), exponential density."""
    nz = case["nz"]
    if case["levels"] == "uniform":
        dz = np.full(nz, min(case["dx"], 20.0))
        return dz, np.ones(nz)
    dz = 10.0 * 1.03 ** np.arange(nz)
    return dz, 1.2 * np.exp(-(np.cumsum(dz) - 0.5 * dz) / 8000.0)


def _noise(gen, shape):
    s = torch.randn(shape, generator=gen, device="cuda", dtype=torch.float64)
    s -= s.mean()
    return s


def _blobs(gen, nz, ny, nx, n=200):
    """200 Gaussian blobs (sigma 2-10 cells, periodic in x and y) and N(0, 0.1) noise, mean removed."""
    u = lambda *k: torch.rand(*k, generator=gen, device="cuda", dtype=torch.float64)  # noqa: E731
    amp = torch.randn(n, generator=gen, device="cuda", dtype=torch.float64)
    sig = 2.0 + 8.0 * u(n)

    def profile(m, periodic):
        d = (torch.arange(m, device="cuda", dtype=torch.float64)[None] - m * u(n)[:, None]).abs()
        d = torch.minimum(d, m - d) if periodic else d
        return torch.exp(-0.5 * (d / sig[:, None]) ** 2)

    gx, gy, gz = profile(nx, True), profile(ny, True), profile(nz, False) * amp[:, None]
    s = 0.1 * torch.randn((nz, ny, nx), generator=gen, device="cuda", dtype=torch.float64)
    for k in range(nz):
        s[k] += (gy * gz[:, k, None]).T @ gx
    s -= s.mean()
    return s


def _source(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    shape = (case["nz"], case["ny"], case["nx"])
    return _blobs(gen, *shape) if case["source"] == "blobs" else _noise(gen, shape)


def _field(x, case):
    """A (nz, ny, nx) double field as the caller of this case holds it."""
    if case.get("layout") == "xyz":
        x = x.permute(2, 1, 0)
    return x.to(torch.float32 if case["dtype"] == "fp32" else torch.float64).contiguous()


def _weights(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed + 7919)
    return torch.randn((case["nz"], case["ny"], case["nx"]), generator=gen, device="cuda", dtype=torch.float64)


def _batch_domains(case):
    """Unequal domains: nx = ny from 64..512, nz from 32..96, seeded spacings, levels and densities."""
    rng = np.random.default_rng(case["shapes"])
    out = []
    for _ in range(case["domains"]):
        n, nz = int(rng.choice([64, 128, 256, 384, 512])), int(rng.choice([32, 48, 64, 96]))
        dx, dz = float(rng.choice([25.0, 50.0, 100.0])), rng.uniform(5.0, 20.0) * rng.uniform(1.0, 1.05) ** np.arange(nz)
        rho = rng.uniform(1.0, 1.3) * np.exp(-(np.cumsum(dz) - 0.5 * dz) / rng.uniform(7000.0, 9000.0))
        out.append((n, nz, dx, dz, rho))
    return out


def _batch_sources(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    dt = torch.float32 if case["dtype"] == "fp32" else torch.float64
    return [_noise(gen, (nz, n, n)).to(dt) for n, nz, _, _, _ in _batch_domains(case)]


def _density3(case, seed):
    """A smooth horizontal perturbation of the level profile (a few long waves, varying slowly in height)."""
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    rng = np.random.default_rng(seed)
    ax = lambda m: torch.arange(m, device="cuda", dtype=torch.float64)  # noqa: E731
    g = torch.zeros((nz, ny, nx), device="cuda", dtype=torch.float64)
    for _ in range(4):
        a, b = int(rng.integers(1, 4)), int(rng.integers(0, 4))
        ph = rng.uniform(0, 2 * np.pi, 3)
        g += (torch.cos(2 * np.pi * a / nx * ax(nx) + ph[0])[None, None, :]
              * torch.cos(2 * np.pi * b / ny * ax(ny) + ph[1])[None, :, None]
              * (1 + 0.5 * torch.cos(np.pi / nz * (ax(nz) + 0.5) + ph[2]))[:, None, None])
    g *= case["perturbation"] / g.abs().max()
    rho0 = torch.from_numpy(_levels(case)[1]).cuda()
    return rho0[:, None, None] * (1 + g)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        doms = [Domain(n, n, nz, dx, dx, dz, rho) for n, nz, dx, dz, rho in _batch_domains(case)]
        S = _batch_sources(case, seed)
        return dict(kind=kind, batch=Batch(doms, dtype=case["dtype"]), S=S, p=[torch.empty_like(s) for s in S])
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    dz, rho = _levels(case)
    if kind == "cg":
        rho3 = _density3(case, seed)
        S = _noise(torch.Generator(device="cuda").manual_seed(seed), (nz, ny, nx))
        # the preconditioner: a plan for the horizontally averaged density
        plan = Plan(nx, ny, nz, case["dx"], case["dy"], dz, rho3.mean(dim=(1, 2)).cpu().numpy(), dtype="mixed",
                    max_sweeps=0)
        return dict(kind=kind, plan=plan, rho3=rho3, S=S, p=torch.empty_like(S))
    S = _field(_source(case, seed), case)
    plan = Plan(nx, ny, nz, case["dx"], case["dy"], dz, rho, dtype=case["dtype"], bc=case.get("bc", "neumann"),
                layout=case.get("layout", "zyx"))
    plan.workspace()
    if kind == "grad":
        rho_t = torch.from_numpy(rho).cuda().requires_grad_() if case["density"] else None
        return dict(kind=kind, plan=plan, S=S.requires_grad_(), rho=rho_t, w=_field(_weights(case, seed), case))
    return dict(kind=kind, plan=plan, S=S, p=torch.empty_like(S))


def run(state):
    kind = state["kind"]
    if kind == "solve":
        return state["plan"].solve(state["S"], out=state["p"])
    if kind == "batch":
        return state["batch"].solve(state["S"], out_list=state["p"])
    if kind == "cg":
        return state["plan"].cg_solve(state["rho3"], state["S"], out=state["p"], tol=1e-10)[0]
    # one training step's use of the projection: p for the loss, then the loss's gradient back through the solve
    p = poisson_solve(state["S"], state["plan"], rho0=state["rho"])
    wrt = (state["S"],) if state["rho"] is None else (state["S"], state["rho"])
    return (p.detach(),) + torch.autograd.grad(p, wrt, grad_outputs=state["w"])


# ---------------------------------------------------------------------------
# the least work of a pass
# ---------------------------------------------------------------------------

def _solve_flops(nx, ny, nz):
    """Real transforms there and back (2.5 n log2 n a line each) and the column elimination (18 a complex entry)."""
    return nx * ny * nz * (5 * math.log2(nx) + 5 * math.log2(ny) + 9)


def work(case):
    kind = case["kind"]
    size = 4 if case.get("dtype") == "fp32" else 8
    if kind == "batch":
        d = _batch_domains(case)
        return {"bytes": sum(2 * size * n * n * nz for n, nz, *_ in d), "flops": sum(_solve_flops(n, n, nz) for n, nz, *_ in d)}
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    n, f = nx * ny * nz, _solve_flops(nx, ny, nz)
    if kind == "cg":   # density and source read, pressure written; a handful of preconditioned iterations
        return {"bytes": 3 * 8 * n, "flops": 8 * (f + 40 * n)}
    if kind == "grad":  # S and w read, p and dL/dS written (p read again for the density gradient)
        return {"bytes": (5 if case["density"] else 4) * size * n, "flops": 2 * f + (10 * n if case["density"] else 0)}
    return {"bytes": 2 * size * n, "flops": f}


# ---------------------------------------------------------------------------
# the same problems in plain torch, 64 bits
# ---------------------------------------------------------------------------

class _Ref:
    """(L p)_k = horizontal second differences + a_k (p_{k-1} - p_k) + c_k (p_{k+1} - p_k)."""

    def __init__(self, nx, ny, nz, dx, dy, dz, rho, lid=False):
        t = lambda v: torch.from_numpy(np.asarray(v, dtype=np.float64)).cuda()  # noqa: E731
        dz, rho = np.asarray(dz, float), np.asarray(rho, float)
        self.W, self.h, self.rf = rho * dz, 0.5 * (dz[1:] + dz[:-1]), 0.5 * (rho[1:] + rho[:-1])
        self.a = np.concatenate([[0.0], self.rf / (self.W[1:] * self.h)])
        self.c = np.concatenate([self.rf / (self.W[:-1] * self.h), [rho[-1] / (self.W[-1] * dz[-1] / 2) if lid else 0.0]])
        self.nx, self.ny, self.nz, self.dx, self.dy, self.rho, self.lid = nx, ny, nz, dx, dy, rho, lid
        kx, ky = np.arange(nx // 2 + 1), np.arange(ny)
        self.s = t(4 / dy ** 2 * np.sin(np.pi * np.minimum(ky, ny - ky) / ny)[:, None] ** 2
                   + 4 / dx ** 2 * np.sin(np.pi * kx / nx)[None, :] ** 2)   # row sums -lambda >= 0

    def solve(self, S):
        """L p = S - mu_W with zero mean (lid: L p = S); S is not kept."""
        F = torch.fft.rfft2(S, dim=(1, 2))
        f0 = F[:, 0, 0].real.cpu().numpy() / (self.nx * self.ny)
        inv = torch.empty((self.nz,) + self.s.shape, device="cuda", dtype=torch.float64)
        g = self.s.clone()
        for k in range(self.nz):     # u_k = s + a_k g_{k-1}/u_{k-1} + c_k: no subtraction, so weak columns keep their digits
            if k:
                g = self.s + self.a[k] * (g * inv[k - 1])
                F[k] += self.a[k] * (F[k - 1] * inv[k - 1])
            u = g + self.c[k]
            if not self.lid:
                u[0, 0] = 1.0        # solved apart below
            inv[k] = 1.0 / u
        F[self.nz - 1] *= -inv[self.nz - 1]
        for k in range(self.nz - 2, -1, -1):
            F[k] = (self.c[k] * F[k + 1] - F[k]) * inv[k]
        if not self.lid:             # the horizontal mean: fluxes summed upwards, then the pressure
            r = f0 - (self.W * f0).sum() / self.W.sum()
            p0 = np.concatenate([[0.0], np.cumsum(np.cumsum(self.W * r)[:-1] * self.h / self.rf)])
            F[:, 0, 0] = torch.from_numpy((p0 - p0.mean()) * self.nx * self.ny).cuda()
        del inv
        return torch.fft.irfft2(F, s=(self.ny, self.nx), dim=(1, 2))

    def adjoint(self, w):
        """G^T w for G = solve (no lid): W L is symmetric, so L^T mu = w - mean(w) for mu = W y, L y = (w - mean)/W."""
        W = torch.from_numpy(self.W).cuda()[:, None, None]
        mu = W * self.solve((w - w.mean()) / W)
        return mu - W * (mu.sum() / (self.W.sum() * self.nx * self.ny))

    def density_gradient(self, mu, p):
        W, h, rf, rho = (torch.from_numpy(v).cuda() for v in (self.W, self.h, self.rf, self.rho))
        D = (p[1:] - p[:-1]) / h[:, None, None]
        y = mu / W[:, None, None]
        flux = (D * (y[:-1] - y[1:])).sum(dim=(1, 2))          # d(-mu^T L p)/d rf, with the sign below
        V = torch.zeros_like(p)
        V[:-1] += rf[:, None, None] * D
        V[1:] -= rf[:, None, None] * D
        out = (y * V).sum(dim=(1, 2)) / rho
        out[:-1] -= 0.5 * flux
        out[1:] -= 0.5 * flux
        return out


def _exact_cg(case, seed):
    nx, ny, nz, dx, dy = (case[k] for k in ("nx", "ny", "nz", "dx", "dy"))
    rho, dz = _density3(case, seed), _levels(case)[0]
    S = _noise(torch.Generator(device="cuda").manual_seed(seed), (nz, ny, nx))
    ref = _Ref(nx, ny, nz, dx, dy, dz, rho.mean(dim=(1, 2)).cpu().numpy())
    t = torch.from_numpy(dz).cuda()[:, None, None]
    W = rho * t
    bx, by = t * (rho + rho.roll(-1, 2)) / (2 * dx * dx), t * (rho + rho.roll(-1, 1)) / (2 * dy * dy)
    bz = (rho[1:] + rho[:-1]) / (t[1:] + t[:-1])
    Wm = torch.from_numpy(ref.W).cuda()[:, None, None]

    def op(p):      # -W A p
        fx, fy, fz = bx * (p.roll(-1, 2) - p), by * (p.roll(-1, 1) - p), bz * (p[1:] - p[:-1])
        q = fx.roll(1, 2) - fx + fy.roll(1, 1) - fy
        q[:-1] -= fz
        q[1:] += fz
        return q

    b = -W * (S - (W * S).sum() / W.sum())
    p, r = torch.zeros_like(b), b
    z = ref.solve(-r / Wm)
    d, rz, first = z, (r * z).sum(), b.norm()
    for _ in range(60):
        q = op(d)
        al = rz / (d * q).sum()
        p, rn = p + al * d, r - al * q
        z = ref.solve(-rn / Wm)
        be = ((rn - r) * z).sum() / rz
        r, rz = rn, (rn * z).sum()
        d = z + be * d
        if r.norm() < 1e-14 * first:
            break
    return p - p.mean()


def exact(case, seed):
    if case["kind"] == "batch":
        return [_Ref(n, n, nz, dx, dx, dz, rho).solve(S.double())
                for (n, nz, dx, dz, rho), S in zip(_batch_domains(case), _batch_sources(case, seed))]
    if case["kind"] == "cg":
        return _exact_cg(case, seed)
    dz, rho = _levels(case)
    ref = _Ref(case["nx"], case["ny"], case["nz"], case["dx"], case["dy"], dz, rho, case.get("bc") == "dirichlet_top")
    rounded = lambda x: x.to(torch.float32 if case["dtype"] == "fp32" else torch.float64).double()  # noqa: E731
    p = ref.solve(rounded(_source(case, seed)))
    if case["kind"] == "solve":
        return p.permute(2, 1, 0).contiguous() if case["layout"] == "xyz" else p
    mu = ref.adjoint(rounded(_weights(case, seed)))
    return (p, mu, ref.density_gradient(mu, p)) if case["density"] else (p, mu)
