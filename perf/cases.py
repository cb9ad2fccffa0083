"""Workloads by which the speed of the library is measured.

A case is a dict of plain values.  Its ``kind`` names the public entry point:

* ``step``      one implicit Euler step of a batch of samples from a state that
                has been marched a few steps from t = 0 (``elder_step``, or
                ``elder_step_predicted`` with the history levels it keeps);
* ``grad``      the discrete adjoint of a short run of one lognormal sample;
* ``residual``  the FP64 residual of a batch;
* ``moments``   mean, variance and exceedance probability over a batch;
* ``project``   the projection of quadrature-point fields on a gPC basis;
* ``exceed``    the exceedance count of a gPC surrogate.

``prepare`` makes what a program holds before the call, ``run`` is one call,
``work`` the bytes of its inputs and outputs and the arithmetic it cannot do
without, ``exact`` the same outputs from plain torch in 64 bits.
"""
from __future__ import annotations

import itertools
import math

import numpy as np
import torch

from paper_1906_01632_gb300 import elder as E
from paper_1906_01632_gb300 import inputs as I

YEAR = E.SECONDS_PER_YEAR
K_MEAN = 4.845e-13
F64 = torch.float64
MOST_COARSE_UNKNOWNS = 200  # of the grids drawn here: those that coarsen far


def _device():
    return torch.device("cuda:0")


def listed():
    return [
        # the first benchmark configuration: one sample on the smallest grid,
        # FP64, Newton from u^n; launches and latency count
        dict(name="step 32x32x8 x1 fp64", kind="step", nx=32, ny=32, nz=8, S=1, mixed=False,
             order=0, bc=0, field=0, dt_yr=1 / 12, warm=2),
        # the paper's 1.1 million unknown mesh, one sample
        dict(name="step 128x128x32 x1 mixed", kind="step", nx=128, ny=128, nz=32, S=1, mixed=True,
             order=2, bc=0, field=0, dt_yr=1 / 12, warm=3),
        # the headline workload: 256 Sobol samples
        dict(name="step 64x64x16 x256 mixed", kind="step", nx=64, ny=64, nz=16, S=256, mixed=True,
             order=2, bc=0, field=0, dt_yr=1 / 12, warm=3),
        # the same method in FP64 throughout, a smaller batch
        dict(name="step 64x64x16 x32 fp64", kind="step", nx=64, ny=64, nz=16, S=32, mixed=False,
             order=2, bc=0, field=0, dt_yr=1 / 12, warm=3),
        # the paper's own ensemble: parallelepiped field at Halton points, its
        # boundary sets and its small time step
        dict(name="step 128x128x32 x24 paper", kind="step", nx=128, ny=128, nz=32, S=24,
             mixed=True, order=2, bc=1, field=2, dt_yr=0.005, warm=3),
        # the large grid of the uneven ensemble
        dict(name="step 256x256x64 x2 mixed", kind="step", nx=256, ny=256, nz=64, S=2, mixed=True,
             order=2, bc=0, field=0, dt_yr=1 / 24, warm=3),
        # an oblong grid, whose coarsening stops at 8 x 4 x 1 cells
        dict(name="step 128x64x16 x4 mixed", kind="step", nx=128, ny=64, nz=16, S=4, mixed=True,
             order=2, bc=0, field=0, dt_yr=1 / 24, warm=2),
        # sensitivities of a lognormal sample (forward, recomputation, adjoint)
        dict(name="grad 64x64x16 4 steps", kind="grad", nx=64, ny=64, nz=16, steps=4, ckpt=2,
             dt_yr=1 / 12),
        # the Newton residual by itself
        dict(name="residual 64x64x16 x64", kind="residual", nx=64, ny=64, nz=16, S=64, bc=0,
             dt_yr=1 / 12),
        # output time of the headline ensemble
        dict(name="moments 64x64x16 x256", kind="moments", nx=64, ny=64, nz=16, S=256,
             weighted=False),
        # the order-4 surrogate of the 5^3 Gauss-Legendre runs
        dict(name="project 125 x 71825, 35 terms", kind="project", M=3, p=4, q=5, N=71825),
        # its exceedance probability at every node
        dict(name="exceed 71825 x 2e5, 35 terms", kind="exceed", M=3, p=4, N=71825, n_pts=0,
             Ns=200_000),
    ]


def _coarse_unknowns(nx, ny, nz, bc):
    """Unknowns of the coarsest grid: counts are halved while all are even and
    (boundary sets 0 and 1) the top square stays on nodes."""
    while not (nx % 2 or ny % 2 or nz % 2):
        if bc in (0, 1) and ((nx // 2) % 4 or (ny // 2) % 4):
            break
        nx, ny, nz = nx // 2, ny // 2, nz // 2
    return 2 * (nx + 1) * (ny + 1) * (nz + 1)


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_grid(rng, bc, most_nodes):
    """A grid of the 600 x 600 x 150 m box with cells of moderate aspect ratio
    that coarsens far."""
    while True:
        nx, ny = (rng.choice((16, 24, 32, 48, 64, 96, 128, 192, 256)) for _ in range(2))
        nz = rng.choice((2, 3, 4, 5, 6, 8, 10, 12, 16, 20, 24, 32, 48, 64))
        N = (nx + 1) * (ny + 1) * (nz + 1)
        if N <= most_nodes and max(nx, ny) <= 2 * min(nx, ny) and \
                max(nx, ny) <= 8 * nz <= 4 * max(nx, ny) and \
                _coarse_unknowns(nx, ny, nz, bc) <= MOST_COARSE_UNKNOWNS:
            return nx, ny, nz, N


def draw(rng):
    kind = rng.choice(("step", "step", "step", "step", "grad", "residual", "moments", "project",
                       "exceed"))
    if kind == "step":
        mixed = rng.random() < 0.7
        bc, field, dt_yr = rng.choice(((0, 0, 1 / 12), (0, 0, 1 / 24), (0, 1, 1 / 24),
                                       (1, 2, 0.005)))
        most = 1_500_000 if not mixed else 600_000 if field == 1 else 6_000_000
        total = _log_int(rng, 9_801, most)
        nx, ny, nz, N = _draw_grid(rng, bc, max(total, 3_000))
        return dict(kind=kind, nx=nx, ny=ny, nz=nz, S=max(1, min(200, total // N)), mixed=mixed,
                    order=rng.choice((0, 1, 2)), bc=bc, field=field, dt_yr=dt_yr,
                    warm=rng.choice((2, 3)))
    if kind == "grad":
        nz = rng.choice((4, 8, 16))
        return dict(kind=kind, nx=4 * nz, ny=4 * nz, nz=nz, steps=rng.choice((2, 3, 4)),
                    ckpt=rng.choice((1, 2, 3)), dt_yr=rng.choice((1 / 12, 1 / 24, 1 / 48)))
    if kind == "residual":
        bc = rng.choice((0, 1, 2, 3))
        step = 4 if bc < 2 else 1
        nx, ny, nz = step * rng.randint(12 // step, 72 // step), step * rng.randint(
            12 // step, 72 // step), rng.randint(3, 20)
        N = (nx + 1) * (ny + 1) * (nz + 1)
        total = _log_int(rng, 10_000, 4_000_000)
        return dict(kind=kind, nx=nx, ny=ny, nz=nz, S=max(1, min(300, total // N)), bc=bc,
                    dt_yr=rng.choice((1 / 12, 1 / 24, 0.005)))
    if kind == "moments":
        nx, ny, nz = 4 * rng.randint(4, 32), 4 * rng.randint(4, 32), rng.randint(4, 32)
        N = (nx + 1) * (ny + 1) * (nz + 1)
        total = _log_int(rng, 100_000, 18_000_000)
        return dict(kind=kind, nx=nx, ny=ny, nz=nz, S=max(2, min(300, total // N)),
                    weighted=rng.random() < 0.5)
    if kind == "project":
        M, p, q = rng.choice(((1, 4, 5), (2, 3, 4), (2, 6, 7), (3, 2, 3), (3, 4, 5), (4, 2, 3),
                              (4, 3, 4)))
        return dict(kind=kind, M=M, p=p, q=q, N=_log_int(rng, 1_000, 150_000))
    M, p = rng.choice(((2, 3), (2, 6), (3, 2), (3, 3), (3, 4), (3, 4), (4, 2), (4, 3)))
    return dict(kind=kind, M=M, p=p, N=_log_int(rng, 1_000, 72_000),
                n_pts=rng.choice((0, 0, rng.randint(100, 1_000))), Ns=_log_int(rng, 2_000, 200_000))


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

def _generator(seed):
    return torch.Generator(device=_device()).manual_seed(int(seed))


def _field_params(case, S, C, seed):
    """(elder_fields kind, parameters): Sobol points of the cosine field, normals
    of the lognormal field, Halton points of the parallelepiped field."""
    field = case.get("field", 1)
    if field == 1:
        return 1, torch.randn(S * C, generator=_generator(seed), dtype=F64, device=_device())
    xi = I.sobol_xi(S, seed=seed) if field == 0 else I.halton_xi(S, skip=1 + seed % 5000)
    return field, torch.tensor(xi.ravel(), dtype=F64, device=_device())


def _prepare_step(case, seed):
    S = case["S"]
    ctx = E.elder_create(E.elder_config_default(
        case["nx"], case["ny"], case["nz"], max_samples=S, bc_mode=case["bc"],
        precision=E.ELDER_MIXED if case["mixed"] else E.ELDER_FP64))
    kind, params = _field_params(case, S, ctx.C, seed)
    phi, K = ctx.fields(S, kind, params, K_mean=K_MEAN)
    p, c = ctx.initial_state(S)
    s = dict(kind="step", ctx=ctx, S=S, phi=phi, K=K, p=p, c=c, dt=case["dt_yr"] * YEAR,
             order=case["order"])
    if s["order"]:
        s["ph"], s["ch"] = p.repeat(s["order"]), c.repeat(s["order"])
    for _ in range(case["warm"]):
        _step(s)
    s["saved"] = [s[k].clone() for k in ("p", "c", "ph", "ch") if k in s]
    return s


def _step(s):
    if s["order"]:
        return s["ctx"].step_predicted(s["S"], s["phi"], s["K"], s["order"], s["ph"], s["ch"],
                                       s["p"], s["c"], s["dt"])
    return s["ctx"].step(s["S"], s["phi"], s["K"], s["p"], s["c"], s["dt"])


def _rough_state(N, S, sxy, nz, seed):
    """A state off equilibrium (upwinding in every direction): hydrostatic
    pressure and a salt fraction in [0, 1], both perturbed node by node."""
    g = _generator(seed)
    k = torch.arange(N, device=_device()) // sxy
    p = (1000.0 * 9.81 * 150.0 * (1.0 - k.to(F64) / nz)).repeat(S)
    p += 2e3 * torch.randn(S * N, generator=g, dtype=F64, device=_device())
    c = torch.rand(S * N, generator=g, dtype=F64, device=_device())
    return p, c


def _plume_fields(n, N, seed):
    """n salt-fraction fields in [0, 1]: a front of random position per field."""
    g = _generator(seed)
    z = torch.linspace(-1.0, 1.0, N, dtype=F64, device=_device())
    at = 0.5 * torch.randn(n, 1, generator=g, dtype=F64, device=_device())
    u = torch.sigmoid(6.0 * (z[None, :] - at))
    u += 0.02 * torch.randn(n, N, generator=g, dtype=F64, device=_device())
    return u.clamp_(0.0, 1.0)


def _rough_inputs(case, seed):
    """Parameters of the lognormal field, state and old state of a residual."""
    S, nz = case["S"], case["nz"]
    sxy = (case["nx"] + 1) * (case["ny"] + 1)
    z = torch.randn(S * case["nx"] * case["ny"] * nz, generator=_generator(seed), dtype=F64,
                    device=_device())
    return (z, *_rough_state(sxy * (nz + 1), S, sxy, nz, seed + 1),
            *_rough_state(sxy * (nz + 1), S, sxy, nz, seed + 2))


def _batch_fields(case, seed):
    """Fields and weights of the sample statistics."""
    N = (case["nx"] + 1) * (case["ny"] + 1) * (case["nz"] + 1)
    w = None
    if case["weighted"]:
        w = torch.rand(case["S"], generator=_generator(seed + 1), dtype=F64, device=_device())
        w /= w.sum()
    return _plume_fields(case["S"], N, seed).reshape(-1), w


def _surrogate(case, seed, degrees):
    """Coefficients of smooth responses (decaying with the degree, means near
    the threshold), node list, points."""
    g, N, dev = _generator(seed), case["N"], _device()
    decay = 0.3 ** torch.tensor(degrees, dtype=F64, device=dev)
    coef = torch.randn(len(degrees), N, generator=g, dtype=F64, device=dev) * decay[:, None]
    coef[0] = 0.3 + 0.4 * torch.rand(N, generator=g, dtype=F64, device=dev)
    nodes = None
    if case["n_pts"]:
        nodes = torch.randperm(N, generator=g, device=dev)[:min(N, case["n_pts"])].to(torch.int32)
    theta = 2.0 * torch.rand(case["Ns"], case["M"], generator=g, dtype=F64, device=dev) - 1.0
    return coef, nodes, theta


def _tensor_rule(M, x, w):
    x, w = torch.tensor(x), torch.tensor(w)
    theta = torch.cartesian_prod(*([x] * M)).reshape(-1, M)
    weight = torch.cartesian_prod(*([w] * M)).reshape(-1, M).prod(1)
    return theta.contiguous().to(_device()), weight.contiguous().to(_device())


def prepare(case, seed):
    kind, dev = case["kind"], _device()
    if kind == "step":
        return _prepare_step(case, seed)
    if kind == "grad":
        ctx = E.elder_create(E.elder_config_default(case["nx"], case["ny"], case["nz"]))
        _, z = _field_params(case, 1, ctx.C, seed)
        phi, K = ctx.fields(1, 1, z, K_mean=K_MEAN)
        p, c = ctx.initial_state(1)
        return dict(kind=kind, ctx=ctx, phi=phi, K=K, p=p, c=c, dt=case["dt_yr"] * YEAR,
                    steps=case["steps"], ckpt=case["ckpt"])
    if kind == "residual":
        S = case["S"]
        ctx = E.elder_create(E.elder_config_default(case["nx"], case["ny"], case["nz"],
                                                    max_samples=S, bc_mode=case["bc"]))
        z, p, c, po, co = _rough_inputs(case, seed)
        phi, K = ctx.fields(S, 1, z, K_mean=K_MEAN)
        return dict(kind=kind, ctx=ctx, S=S, phi=phi, K=K, p=p, c=c, po=po, co=co,
                    dt=case["dt_yr"] * YEAR, R=torch.empty(2 * S * ctx.N, dtype=F64, device=dev))
    if kind == "moments":
        # (workspace for one sample: the statistics take any number of fields)
        ctx = E.elder_create(E.elder_config_default(case["nx"], case["ny"], case["nz"],
                                                    bc_mode=2))
        c, w = _batch_fields(case, seed)
        return dict(kind=kind, ctx=ctx, S=case["S"], w=w, c=c)
    beta = E.elder_gpc_indices(case["M"], case["p"])
    if kind == "project":
        theta, w = _tensor_rule(case["M"], *E.elder_gauss_legendre(case["q"]))
        return dict(kind=kind, beta=torch.tensor(beta, device=dev), theta=theta, w=w,
                    u=_plume_fields(theta.shape[0], case["N"], seed))
    coef, nodes, theta = _surrogate(case, seed, beta.sum(1))
    return dict(kind=kind, beta=torch.tensor(beta, device=dev), coef=coef, theta=theta,
                nodes=nodes)


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------

def run(state):
    s = state
    kind = s["kind"]
    if kind == "step":
        # the same step again: a run restarted from its saved state
        for k, v in zip(("p", "c", "ph", "ch"), s["saved"]):
            s[k].copy_(v)
        status, stats = _step(s)
        out = {"p": s["p"], "c": s["c"], "status": status,
               "salt_mass": [x["salt_mass"] for x in stats[:16]]}
        if s["order"]:
            out["p_hist"], out["c_hist"] = s["ph"], s["ch"]
        return out
    if kind == "grad":
        J, gphi, gK = s["ctx"].grad(s["steps"], s["phi"], s["K"], s["p"], s["c"], s["dt"],
                                    s["ckpt"])
        return {"J": J, "dphi": gphi, "dK": gK}
    if kind == "residual":
        return s["ctx"].residual(s["S"], s["phi"], s["K"], s["p"], s["c"], s["po"], s["co"],
                                 s["dt"], R=s["R"])
    if kind == "moments":
        return s["ctx"].moments(s["S"], s["c"], w=s["w"], threshold=0.5)
    if kind == "project":
        return E.elder_gpc_project(s["beta"], s["theta"], s["w"], s["u"])
    return E.elder_gpc_exceed(s["beta"], s["coef"], s["theta"], 0.5, s["nodes"])


def work(case):
    kind = case["kind"]
    if kind in ("step", "grad", "residual", "moments"):
        N = (case["nx"] + 1) * (case["ny"] + 1) * (case["nz"] + 1)
        C = case["nx"] * case["ny"] * case["nz"]
    res = 340  # flops per node of one evaluation of the discrete equations
    if kind == "step":
        # fields, state and history in, state and history out; the equations
        # hold at the new state: evaluated at least there and at the start
        S, levels = case["S"], 1 + case["order"]
        return {"bytes": 8.0 * S * (2 * C + 4 * levels * N), "flops": 2.0 * res * S * N}
    if kind == "grad":
        # every step forward, and its transposed linearisation once
        n = case["steps"]
        return {"bytes": 8.0 * (4 * C + 2 * N + 4 * n * N), "flops": 4.0 * res * n * N}
    if kind == "residual":
        S = case["S"]
        return {"bytes": 8.0 * S * (2 * C + 5 * N), "flops": float(res * S * N)}
    if kind == "moments":
        return {"bytes": 8.0 * N * (case["S"] + 3), "flops": 6.0 * N * case["S"]}
    T = math.comb(case["M"] + case["p"], case["p"])
    if kind == "project":
        Nq, N = case["q"] ** case["M"], case["N"]
        return {"bytes": 8.0 * N * (Nq + T + 2), "flops": 2.0 * N * Nq * T}
    n = min(case["N"], case["n_pts"]) or case["N"]
    return {"bytes": 8.0 * (n * (T + 1) + case["Ns"] * case["M"]),
            "flops": 2.0 * n * T * case["Ns"]}


# ---------------------------------------------------------------------------
# the same outputs in plain 64-bit torch
# ---------------------------------------------------------------------------

RHO0, DRHO, MU, GRAV, DM = 1000.0, 200.0, 1e-3, 9.81, 3.565e-6
LX, LY, LZ = 600.0, 600.0, 150.0


def _kozeny_carman(phi):
    return K_MEAN * (phi ** 3 / (1.0 - phi) ** 2) / (0.1 ** 3 / 0.9 ** 2)


def _exact_fields(kind, params, S, nx, ny, nz):
    dev = params.device
    x = (torch.arange(nx, dtype=F64, device=dev) + 0.5) * (LX / nx)
    y = (torch.arange(ny, dtype=F64, device=dev)[:, None] + 0.5) * (LY / ny)
    z = (torch.arange(nz, dtype=F64, device=dev)[:, None, None] + 0.5) * (LZ / nz)
    if kind == 1:
        phi = (0.1 * torch.exp(0.2 * params)).clamp(0.05, 0.2).reshape(S, nz, ny, nx)
    else:
        a, b, d = (params.reshape(S, 3)[:, i, None, None, None] for i in range(3))
        if kind == 0:
            phi = 0.1 * (1.0 + 0.1 * (a * torch.cos(math.pi * x / LX) + b * torch.cos(
                math.pi * y / LY) + d * torch.sin(2.0 * math.pi * z / LZ)))
        else:
            sx, sy, sz = (torch.sin(math.pi * x / LX), torch.sin(math.pi * y / LY),
                          torch.sin(math.pi * z / LZ))
            phi = 0.1 + 0.01 * (a * sx + b * sy + d * sz + a * sx * sy + b * sx * sz)
        phi = phi.expand(S, nz, ny, nx)
    return phi, _kozeny_carman(phi)


def _dirichlet(nx, ny, nz, bc, dev):
    """Masks of the p and c Dirichlet nodes and the c values, [nz+1][ny+1][nx+1]."""
    i = torch.arange(nx + 1, device=dev).expand(nz + 1, ny + 1, nx + 1)
    j = torch.arange(ny + 1, device=dev)[:, None].expand_as(i)
    k = torch.arange(nz + 1, device=dev)[:, None, None].expand_as(i)
    top, bottom = k == nz, k == 0
    xe, ye = (i == 0) | (i == nx), (j == 0) | (j == ny)
    sq = (4 * i >= nx) & (4 * i <= 3 * nx) & (4 * j >= ny) & (4 * j <= 3 * ny)
    if bc == 0:
        return top & xe & ye, (top & sq) | bottom, (top & sq).to(F64)
    if bc == 1:
        return top & (xe | ye), top | bottom, (top & sq).to(F64)
    if bc == 2:
        return top & xe & ye, top | bottom, top.to(F64)
    return top & xe & ye, torch.zeros_like(top), torch.zeros_like(top, dtype=F64)


def _corner(u, lx, ly, lz):
    """Values of a node field at one corner of every cell."""
    nz, ny, nx = (n - 1 for n in u.shape[-3:])
    return u[..., lz:lz + nz, ly:ly + ny, lx:lx + nx]


def _pad_corner(f, lx, ly, lz):
    """A cell field added onto the nodes at one of the cells' corners."""
    return torch.nn.functional.pad(f, (lx, 1 - lx, ly, 1 - ly, lz, 1 - lz))


def _exact_residual(p, c, c_old, phi, K, dt, bc, dirichlet):
    """(R_p, R_c) of the box method on [..., nz+1, ny+1, nx+1] node fields."""
    nz, ny, nx = phi.shape[-3:]
    h = (LX / nx, LY / ny, LZ / nz)
    vol = h[0] * h[1] * h[2] / 8.0
    rho_n, rho_o = RHO0 + DRHO * c, RHO0 + DRHO * c_old
    phis = sum(_pad_corner(phi, a, b, d) for a in (0, 1) for b in (0, 1) for d in (0, 1))
    Rp = phis * vol / dt * (rho_n - rho_o)
    Rc = phis * vol / dt * (rho_n * c - rho_o * c_old)
    for D in range(3):
        area = 0.25 * h[(D + 1) % 3] * h[(D + 2) % 3]
        others = [a for a in range(3) if a != D]

        def at(u, v, end):
            at_ = [0, 0, 0]
            at_[D], at_[others[0]], at_[others[1]] = end, u, v
            return at_

        for S_ in (0, 1):
            for T_ in (0, 1):
                gp = gc = ci = 0.0
                for u in (0, 1):
                    for v in (0, 1):
                        w = (0.75 if u == S_ else 0.25) * (0.75 if v == T_ else 0.25)
                        A, B = at(u, v, 0), at(u, v, 1)
                        gp = gp + w * (_corner(p, *B) - _corner(p, *A))
                        gc = gc + w * (_corner(c, *B) - _corner(c, *A))
                        ci = ci + 0.5 * w * (_corner(c, *A) + _corner(c, *B))
                rho = RHO0 + DRHO * ci
                drive = gp / h[D] + (GRAV * rho if D == 2 else 0.0)
                m = -rho * (K / MU) * drive * area
                A, B = at(S_, T_, 0), at(S_, T_, 1)
                up = torch.where(m >= 0.0, _corner(c, *A), _corner(c, *B))
                F = up * m - rho * phi * DM * area * gc / h[D]
                Rp = Rp + _pad_corner(m, *A) - _pad_corner(m, *B)
                Rc = Rc + _pad_corner(F, *A) - _pad_corner(F, *B)
    on_p, on_c, c_d = dirichlet
    return torch.where(on_p, p, Rp), torch.where(on_c, c - c_d, Rc)


def _stencil(f, u):
    """Jacobian of the residual f at u [2, nz+1, ny+1, nx+1] as blocks
    [27][row component][column component][nz+1, ny+1, nx+1]: one directional
    derivative per class of nodes three apart."""
    _, nk, nj, ni = u.shape
    dev = u.device
    k = torch.arange(nk, device=dev)[:, None, None]
    j = torch.arange(nj, device=dev)[:, None]
    i = torch.arange(ni, device=dev)
    colour = (i % 3 + 3 * (j % 3) + 9 * (k % 3)).expand(nk, nj, ni)
    V = torch.zeros(54, 2, nk, nj, ni, dtype=F64, device=dev)
    for q in range(27):
        V[2 * q, 0] = V[2 * q + 1, 1] = (colour == q).to(F64)
    JV = torch.func.vmap(lambda v: torch.func.jvp(f, (u,), (v,))[1])(V)
    J = torch.zeros(27, 2, 2, nk, nj, ni, dtype=F64, device=dev)
    for dz in (-1, 0, 1):
        for dy in (-1, 0, 1):
            for dx in (-1, 0, 1):
                there = ((i + dx) % 3 + 3 * ((j + dy) % 3) + 9 * ((k + dz) % 3)).expand(nk, nj, ni)
                inside = ((i + dx >= 0) & (i + dx < ni) & (j + dy >= 0) & (j + dy < nj) &
                          (k + dz >= 0) & (k + dz < nk)).expand(nk, nj, ni)
                for col in (0, 1):
                    for row in (0, 1):
                        v = torch.gather(JV[:, row], 0, (2 * there + col)[None])[0]
                        J[dx + 1 + 3 * (dy + 1) + 9 * (dz + 1), row, col] = torch.where(
                            inside, v, torch.zeros_like(v))
    return J


def _plane_blocks(J):
    """The blocks coupling x-plane i with planes i - 1, i, i + 1: [3][ni][n][n],
    n the unknowns of a plane."""
    _, _, _, nk, nj, ni = J.shape
    dev, n = J.device, 2 * nk * nj
    out = torch.zeros(3, ni, n, n, dtype=F64, device=dev)
    node = torch.arange(nk * nj, device=dev).reshape(nk, nj)
    for dz in (-1, 0, 1):
        for dy in (-1, 0, 1):
            k = slice(max(0, -dz), nk - max(0, dz))
            j = slice(max(0, -dy), nj - max(0, dy))
            rows, cols = node[k, j].reshape(-1), node[k, j].reshape(-1) + dy + nj * dz
            for dx in (-1, 0, 1):
                b = J[dx + 1 + 3 * (dy + 1) + 9 * (dz + 1)]
                for r in (0, 1):
                    for q in (0, 1):
                        out[dx + 1][:, 2 * rows + r, 2 * cols + q] = \
                            b[r, q][k, j].reshape(-1, ni).T
    return out


def _block_solve(blocks, rhs):
    """Block tridiagonal elimination along x; rhs [ni][n]."""
    lower, diag, upper = blocks
    ni = rhs.shape[0]
    G, y = [], []
    for i in range(ni):
        D, b = diag[i], rhs[i]
        if i:
            D = D - lower[i] @ G[-1]
            b = b - lower[i] @ y[-1]
        full = torch.linalg.solve(D, torch.cat([upper[i], b[:, None]], 1))
        G.append(full[:, :-1])
        y.append(full[:, -1])
    x = [y[-1]]
    for i in range(ni - 2, -1, -1):
        x.insert(0, y[i] - G[i] @ x[0])
    return torch.stack(x)


def _exact_step(p, c, phi, K, dt, bc, dirichlet):
    on_p, on_c, c_d = dirichlet
    c_old = c
    u = torch.stack([torch.where(on_p, torch.zeros_like(p), p), torch.where(on_c, c_d, c)])

    def f(v):
        return torch.stack(_exact_residual(v[0], v[1], c_old, phi, K, dt, bc, dirichlet))

    _, nk, nj, ni = u.shape
    scale = torch.tensor([RHO0 * GRAV * LZ, 1.0], dtype=F64, device=u.device)
    R = f(u)
    for _ in range(40):
        rhs = -R.permute(3, 1, 2, 0).reshape(ni, -1)
        d = _block_solve(_plane_blocks(_stencil(f, u)), rhs).reshape(ni, nk, nj, 2)
        d = d.permute(3, 1, 2, 0)
        small = bool((d.abs().amax((1, 2, 3)) < 1e-13 * scale).all())
        lam = 1.0
        trial = f(u + d)
        while not small and lam > 1e-3 and not trial.norm() < (1.0 - 1e-4 * lam) * R.norm():
            if bool((lam * d.abs().amax((1, 2, 3)) < 1e-11 * scale).all()):
                break
            lam *= 0.5
            trial = f(u + lam * d)
        u, R = u + lam * d, trial
        if small:
            break
    return u[0], u[1]


def _exact_run_of_steps(case, seed):
    nx, ny, nz, S, bc = (case[k] for k in ("nx", "ny", "nz", "S", "bc"))
    dev, dt = _device(), case["dt_yr"] * YEAR
    kind, params = _field_params(case, S, nx * ny * nz, seed)
    phi, K = _exact_fields(kind, params, S, nx, ny, nz)
    dirichlet = _dirichlet(nx, ny, nz, bc, dev)
    z = torch.arange(nz + 1, dtype=F64, device=dev)[:, None, None] * (LZ / nz)
    p0 = (RHO0 * GRAV * (LZ - z)).expand(nz + 1, ny + 1, nx + 1)
    levels, mass = [], []
    for s in range(S):
        us = [(p0, dirichlet[2])]
        for _ in range(case["warm"] + 1):
            us.append(_exact_step(*us[-1], phi[s], K[s], dt, bc, dirichlet))
        us = [us[0]] * 2 + us
        levels.append(us[::-1])
        c = us[-1][1]
        phis = sum(_pad_corner(phi[s], a, b, d) for a in (0, 1) for b in (0, 1) for d in (0, 1))
        vol = LX * LY * LZ / (8.0 * nx * ny * nz)
        mass.append(float((phis * vol * (RHO0 + DRHO * c) * c).sum()))

    def field(level, comp):
        return torch.stack([us[level][comp].reshape(-1) for us in levels]).reshape(-1)

    out = {"p": field(0, 0), "c": field(0, 1), "status": None, "salt_mass": mass[:16]}
    if case["order"]:
        for k, comp in (("p_hist", 0), ("c_hist", 1)):
            out[k] = torch.cat([field(1 + q, comp) for q in range(case["order"])])
    return out


def _legendre(n, x):
    P = [torch.ones_like(x), x]
    for k in range(1, n):
        P.append(((2 * k + 1) * x * P[k] - k * P[k - 1]) / (k + 1))
    return P


def _basis(beta, theta):
    P = [_legendre(max(1, max(row[m] for row in beta)), theta[:, m])
         for m in range(theta.shape[1])]
    return torch.stack([math.prod(P[m][b] for m, b in enumerate(row)) for row in beta])


def _multi_indices(M, p):
    """Total degree at most p, by degree, then lexicographically."""
    every = [b for b in itertools.product(range(p + 1), repeat=M) if sum(b) <= p]
    return sorted(every, key=lambda b: (sum(b), b))


def exact(case, seed):
    kind = case["kind"]
    if kind == "step":
        N = (case["nx"] + 1) * (case["ny"] + 1) * (case["nz"] + 1)
        plane = 2 * (case["ny"] + 1) * (case["nz"] + 1)
        if case["S"] * N > 10_000 or plane > 600:
            return None
        return _exact_run_of_steps(case, seed)
    if kind == "grad":
        return None
    if kind == "residual":
        nx, ny, nz, S, bc = (case[k] for k in ("nx", "ny", "nz", "S", "bc"))
        z, p, c, _, co = _rough_inputs(case, seed)
        phi, K = _exact_fields(1, z, S, nx, ny, nz)
        p, c, co = (v.reshape(S, nz + 1, ny + 1, nx + 1) for v in (p, c, co))
        R = _exact_residual(p, c, co, phi, K, case["dt_yr"] * YEAR, bc,
                            _dirichlet(nx, ny, nz, bc, _device()))
        return torch.stack(R, -1).reshape(-1)
    if kind == "moments":
        S = case["S"]
        c, w = _batch_fields(case, seed)
        c = c.reshape(S, -1)
        w = w if w is not None else torch.full((S,), 1.0 / S, dtype=F64, device=_device())
        mean = w @ c
        return mean, w @ (mean - c) ** 2, w @ (c > 0.5).to(F64)
    beta = _multi_indices(case["M"], case["p"])
    if kind == "project":
        theta, w = _tensor_rule(case["M"], *np.polynomial.legendre.leggauss(case["q"]))
        Q = torch.tensor([math.prod(1.0 / (2 * b + 1) for b in row) for row in beta], dtype=F64,
                         device=_device())
        u = _plume_fields(theta.shape[0], case["N"], seed)
        coef = (0.5 ** case["M"] / Q)[:, None] * ((_basis(beta, theta) * w) @ u)
        return coef, coef[0], (Q[1:, None] * coef[1:] ** 2).sum(0)
    coef, nodes, theta = _surrogate(case, seed, [sum(row) for row in beta])
    coef = coef if nodes is None else coef[:, nodes.long()]
    count = torch.zeros(coef.shape[1], dtype=F64, device=_device())
    for b in _basis(beta, theta).split(4096, dim=1):
        count += (coef.T @ b > 0.5).sum(1)
    return count / case["Ns"]
