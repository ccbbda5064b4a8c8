"""The work that users of this solver have it do, as timed cases.

Every case goes through the public entry points (fv.Solver, the autograd
functions, the surrogate network's train and predict) on states of the kinds
the solver is used on: the isentropic vortex, the Kelvin-Helmholtz layer, the
Taylor-Green vortex, rotated Sod problems and smooth states with noise.  Sizes
run from grids that one SM could hold to the 4096^2 and 384^3 grids of the
benchmark, even and odd, periodic and transmissive.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2306_14011_gb300 import fv
from paper_2306_14011_gb300 import inputs as I
from paper_2306_14011_gb300.autograd import FvRunFunction, kinetic_energy

GAMMA = 1.4
# Operations of one cell and RK stage, every +, -, *, / and sqrt of the plain
# method one operation (as python -m oracle.count_flops counts them).
FLOP_CELL_STAGE = {2: 496.44, 3: 959.62}


def listed():
    return [
        # A residual with its norms on the small grid a solver is debugged and
        # monitored on: latency and launches.
        dict(name="residual_128", kind="residual", ic="vortex", dim=2, nx=128, ny=128, nz=1, bc="periodic",
             limiter="minmod", recon="conserved"),
        # The basic run: isentropic vortex, 128 x 128, 100 steps at CFL 0.5.
        dict(name="run_vortex_128", kind="run", ic="vortex", dim=2, nx=128, ny=128, nz=1, bc="periodic",
             limiter="minmod", recon="conserved", steps=100, source=False),
        # An ordinary grid that no tile divides, shocks, open boundaries, the
        # van Leer limiter on primitive variables.
        dict(name="run_sod_1021x767", kind="run", ic="sod", dim=2, nx=1021, ny=767, nz=1, bc="transmissive",
             limiter="vanleer", recon="primitive", steps=4, source=False),
        # The headline size: Kelvin-Helmholtz on 4096 x 4096.
        dict(name="run_kh_4096", kind="run", ic="kh", dim=2, nx=4096, ny=4096, nz=1, bc="periodic",
             limiter="minmod", recon="conserved", steps=2, source=False),
        # A small ragged box in 3D with open ends along z and a source term.
        dict(name="run_3d_97x66x51", kind="run", ic="smooth", dim=3, nx=97, ny=66, nz=51, bc="mixed",
             limiter="minmod", recon="conserved", steps=4, source=True),
        # The 3D benchmark: Taylor-Green on 384^3, one step.
        dict(name="run_tgv_384", kind="run", ic="tgv", dim=3, nx=384, ny=384, nz=384, bc="periodic",
             limiter="minmod", recon="conserved", steps=1, source=False),
        # Many independent grids of uneven sizes in one call.
        dict(name="batch_sod_96", kind="batch", count=96, nmin=64, nmax=2048, sizes_seed=3, steps=2),
        # One vector-Jacobian product of the residual, on the vortex the adjoint
        # is used on.
        dict(name="vjp_vortex_1024", kind="vjp", ic="vortex", dim=2, nx=1024, ny=1024, nz=1, bc="periodic"),
        # The reverse of one 3D time step.
        dict(name="step_vjp_3d_96", kind="step_vjp", ic="smooth", dim=3, nx=96, ny=96, nz=96, bc="periodic"),
        # A gradient through a checkpointed run, as an optimiser calls it.
        dict(name="grad_vortex_256", kind="grad", ic="vortex", dim=2, nx=256, ny=256, nz=1, bc="periodic", steps=40,
             every=20),
        # A host program that keeps its state in page-locked host memory and
        # advances it one step per call.
        dict(name="host_kh_2048", kind="host_run", ic="kh", dim=2, nx=2048, ny=2048, nz=1, steps=1),
        # One round of the autotuner's surrogate: train on the timed launches,
        # score the random candidates.
        dict(name="surrogate_750_200k", kind="surrogate", features=14, train=750, epochs=20, candidates=200000),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["residual", "run", "run", "run", "batch", "vjp", "step_vjp", "grad", "host_run", "surrogate"])
    dim = rng.choice([2, 2, 3])
    if kind == "surrogate":
        return dict(kind=kind, features=rng.choice([14, 20]), train=_log_int(rng, 200, 1500), epochs=rng.randint(5, 25),
                    candidates=_log_int(rng, 10000, 400000))
    if kind == "batch":
        return dict(kind=kind, count=rng.randint(8, 96), nmin=64, nmax=_log_int(rng, 128, 2048),
                    sizes_seed=rng.randint(0, 10 ** 6), steps=rng.randint(1, 2))
    if kind == "host_run":
        n = _log_int(rng, 256, 4096)
        return dict(kind=kind, ic="kh", dim=2, nx=n, ny=n, nz=1, steps=rng.randint(1, 2))
    if kind == "grad":
        n = _log_int(rng, 96, 512)
        return dict(kind=kind, ic="vortex", dim=2, nx=n, ny=n, nz=1, bc="periodic", steps=rng.randint(10, 60),
                    every=rng.randint(5, 25))
    hi = {"residual": 4096, "run": 4096, "vjp": 2048, "step_vjp": 2048}[kind]
    lo = 48
    if dim == 2:
        nx = _log_int(rng, lo, hi)
        ny = max(lo, min(hi, int(round(nx * math.exp(rng.uniform(-0.7, 0.7))))))
        nz = 1
        ic = rng.choice(["vortex", "kh", "sod", "smooth"])
    else:
        hi = {"residual": 288, "run": 288, "vjp": 160, "step_vjp": 128}[kind]
        nx = _log_int(rng, 24, hi)
        ny = max(16, min(hi, int(round(nx * math.exp(rng.uniform(-0.5, 0.5))))))
        nz = max(16, min(hi, int(round(nx * math.exp(rng.uniform(-0.5, 0.5))))))
        ic = rng.choice(["tgv", "smooth"])
    bc = "transmissive" if ic == "sod" else rng.choice(["periodic", "mixed"] if ic == "smooth" else ["periodic"])
    c = dict(kind=kind, ic=ic, dim=dim, nx=nx, ny=ny, nz=nz, bc=bc)
    if kind in ("residual", "run"):
        # minmod on the conserved variables is what most users run
        c["limiter"] = rng.choice(["minmod", "minmod", "minmod", "vanleer", "none"])
        c["recon"] = rng.choice(["conserved", "conserved", "conserved", "primitive"])
    if kind == "run":
        cells = nx * ny * nz * (2 if dim == 3 else 1)
        c["steps"] = max(1, min(100, int(rng.uniform(0.2, 1.0) * 2 * 4096 * 4096 / cells)))
        c["source"] = rng.random() < 0.2
    return c


# ----------------------------------------------------------------------------- inputs, made on the GPU

def _grid(case):
    d = case["dim"]
    P, T = I.BC_PERIODIC, I.BC_TRANSMISSIVE
    bc = {"periodic": ((P, P), (P, P), (P, P)), "transmissive": ((T, T), (T, T), (T, T)),
          "mixed": ((P, P), (P, P), (T, T)) if d == 3 else ((P, P), (T, T), (P, P))}[case.get("bc", "periodic")]
    if d == 2:
        bc = (bc[0], bc[1], (P, P))
    n = (case["nx"], case["ny"], case["nz"])
    L = {"vortex": 10.0, "kh": 1.0, "sod": 1.0, "smooth": 1.0, "tgv": 2.0 * math.pi}[case["ic"]]
    return I.GridSpec(d, n, (L, L, L if d == 3 else 1.0), bc)


def _conserved(rho, vel, p):
    U = torch.empty((len(vel) + 2,) + tuple(rho.shape), dtype=torch.float64, device=rho.device)
    U[0] = rho
    ke = torch.zeros_like(rho)
    for d, v in enumerate(vel):
        U[1 + d] = rho * v
        ke += v * v
    U[-1] = p / (GAMMA - 1.0) + 0.5 * rho * ke
    return U


def _centres(g, dev):
    h = g.spacing
    return [(torch.arange(g.n[d], dtype=torch.float64, device=dev) + 0.5) * h[d] for d in range(g.dim)]


def _state(case, g, seed):
    """The initial states of paper_2306_14011_gb300/inputs.py, formed on the GPU from the seed."""
    dev = torch.device("cuda")
    gen = torch.Generator(device=dev)
    gen.manual_seed(seed)
    rng = np.random.default_rng(seed)

    def noise(shape):
        return 2.0 * torch.rand(shape, dtype=torch.float64, device=dev, generator=gen) - 1.0

    cc = _centres(g, dev)
    shape = g.shape[1:]
    ic = case["ic"]
    if ic == "vortex":
        x, y = cc[0][None, :], cc[1][:, None]
        dx, dy = x - 5.0, y - 5.0
        r2 = dx * dx + dy * dy
        amp = 5.0 / (2.0 * math.pi) * torch.exp(0.5 * (1.0 - r2))
        u = 0.5 * math.sqrt(GAMMA) - amp * dy
        v = amp * dx
        T = 1.0 - (GAMMA - 1.0) * 25.0 / (8.0 * GAMMA * math.pi ** 2) * torch.exp(1.0 - r2)
        rho = T ** (1.0 / (GAMMA - 1.0))
        return _conserved(rho + 1e-3 * noise(shape), (u, v), rho ** GAMMA)
    if ic == "kh":
        x, y = cc[0], cc[1]
        phi = rng.random(8) * 2.0 * math.pi
        sx = sum(torch.sin(2.0 * math.pi * m * x + phi[m - 1]) for m in range(1, 9)) * (0.01 / 8)
        gy = torch.exp(-((y - 0.25) ** 2) / 0.005) + torch.exp(-((y - 0.75) ** 2) / 0.005)
        band = ((y - 0.5).abs() < 0.25)[:, None].expand(shape)
        one = torch.ones(shape, dtype=torch.float64, device=dev)
        return _conserved(torch.where(band, 2.0 * one, one), (torch.where(band, 0.5 * one, -0.5 * one),
                                                              gy[:, None] * sx[None, :]), 2.5 * one)
    if ic == "sod":
        th = rng.uniform(0.0, 2.0 * math.pi)
        left = (cc[0][None, :] - 0.5) * math.cos(th) + (cc[1][:, None] - 0.5) * math.sin(th) < 0.0
        one = torch.ones(shape, dtype=torch.float64, device=dev)
        return _conserved(torch.where(left, one, 0.125 * one), (0.0 * one, 0.0 * one), torch.where(left, one, 0.1 * one))
    if ic == "tgv":
        x, y, z = cc[0][None, None, :], cc[1][None, :, None], cc[2][:, None, None]
        u = torch.sin(x) * torch.cos(y) * torch.cos(z)
        v = -torch.cos(x) * torch.sin(y) * torch.cos(z)
        p = 1.0 / (GAMMA * 0.01) + (torch.cos(2 * x) + torch.cos(2 * y)) * (torch.cos(2 * z) + 2.0) / 16.0
        p = p * (1.0 + 1e-4 * noise(shape))
        return _conserved(torch.ones_like(p), (u, v, torch.zeros_like(p)), p)
    # smooth: a few random Fourier modes and white noise around a mean flow
    axes = [c.reshape([-1 if g.dim - 1 - d == a else 1 for a in range(g.dim)]) for d, c in enumerate(cc)]

    def field(base):
        f = torch.full(shape, base, dtype=torch.float64, device=dev)
        for _ in range(3):
            k = rng.integers(1, 4, size=g.dim)
            f = f + 0.2 / 3.0 * torch.sin(rng.random() * 2 * math.pi
                                          + sum(2 * math.pi * int(k[d]) / g.length[d] * axes[d] for d in range(g.dim)))
        return f + 1e-3 * noise(shape)

    rho, p = field(1.0), field(1.0)
    return _conserved(rho, tuple(field(b) for b in (0.3, -0.2, 0.1)[:g.dim]), p)


def _source(g, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed + 7)
    return 0.1 * torch.randn(g.shape, dtype=torch.float64, device="cuda", generator=gen)


def _cotangent(g, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed + 5)
    return torch.randn(g.shape, dtype=torch.float64, device="cuda", generator=gen)


def _batch_states(case, seed):
    sizes = [n for n, _ in I.batched_sod(case["count"], case["sizes_seed"], case["nmin"], case["nmax"])]
    cs = [dict(ic="sod", dim=2, nx=n, ny=n, nz=1, bc="transmissive") for n in sizes]
    grids = [_grid(c) for c in cs]
    return grids, [_state(c, g, seed + i) for i, (c, g) in enumerate(zip(cs, grids))]


LIMITER = {"minmod": fv.FV_LIM_MINMOD, "vanleer": fv.FV_LIM_VANLEER, "none": fv.FV_LIM_NONE}
RECON = {"conserved": fv.FV_RECON_CONSERVED, "primitive": fv.FV_RECON_PRIMITIVE}


def _surrogate_data(case, seed):
    sizes = [case["features"], 128, 64, 32, 1]
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)

    def rand(*s):
        return torch.rand(s, dtype=torch.float64, device="cuda", generator=gen)

    def features(rows):  # log2 of launch parameters on their value sets, standardised
        return (torch.floor(5.0 * rand(rows, case["features"])) - 2.0) / math.sqrt(2.0)

    X = features(case["train"])
    y = torch.tanh(X[:, 0] - 0.5 * X[:, 1]) + 0.3 * X[:, 2] * X[:, 3] + 0.05 * (2.0 * rand(case["train"]) - 1.0)
    parts = []
    for fi, fo in zip(sizes[:-1], sizes[1:]):
        bound = math.sqrt(6.0 / (fi + fo))
        parts += [(2.0 * rand(fi * fo) - 1.0) * bound, (2.0 * rand(fo) - 1.0) * bound]
    order = torch.stack([torch.randperm(case["train"], device="cuda", generator=gen) for _ in range(case["epochs"])])
    return sizes, torch.cat(parts), X, y, order.to(torch.int32), features(case["candidates"])


def prepare(case, seed):
    kind = case["kind"]
    if kind == "surrogate":
        sizes, params, X, y, order, C = _surrogate_data(case, seed)
        return dict(case=case, sizes=sizes, params0=params, params=params.clone(), X=X, y=y, order=order, C=C,
                    scores=torch.empty(case["candidates"], dtype=torch.float64, device="cuda"),
                    hyper=fv.mlp_hyper(n_iter_no_change=0))
    if kind == "batch":
        grids, states = _batch_states(case, seed)
        s = fv.Solver(grids)
        U0 = s.pack(states)
        return dict(case=case, solver=s, U0=U0, U=U0.clone())
    g = _grid(case)
    U0 = _state(case, g, seed)
    s = fv.Solver(g, limiter=LIMITER[case.get("limiter", "minmod")], recon=RECON[case.get("recon", "conserved")])
    st = dict(case=case, solver=s, grid=g, U0=U0)
    if kind == "run":
        st["U"] = U0.clone()
        if case["source"]:
            s.set_source(_source(g, seed))
    elif kind == "residual":
        st["R"] = torch.empty_like(U0)
    elif kind == "host_run":
        h = torch.empty(g.shape, dtype=torch.float64, pin_memory=True)
        h.copy_(U0)
        st["pinned"], st["host"] = h, h.numpy()
        del st["U0"]
    else:
        st["lam"] = _cotangent(g, seed)
        st["out"] = torch.empty_like(U0)
        st["dt"] = s.time_step(U0)
    return st


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "surrogate":
        state["params"].copy_(state["params0"])
        losses = fv.fv_mlp_train(state["sizes"], state["params"], state["X"], state["y"], state["order"], state["hyper"])
        fv.fv_mlp_predict(state["sizes"], state["params"], state["C"], state["scores"])
        return {"params": state["params"], "scores": state["scores"], "losses": np.array(losses)}
    s = state["solver"]
    if kind == "residual":
        R, norms = s.residual(state["U0"], state["R"], norms=True)
        return {"R": R, "norms": norms}
    if kind in ("run", "batch"):
        state["U"].copy_(state["U0"])
        s.run(state["U"], case["steps"])
        return {"U": state["U"]}
    if kind == "host_run":
        s.run(state["host"], case["steps"])
        return {"U": state["host"]}
    if kind == "vjp":
        return {"g": s.residual_vjp(state["U0"], state["lam"], state["out"])}
    if kind == "step_vjp":
        return {"g": s.rk_step_vjp(state["U0"], state["lam"], state["dt"], state["out"])}
    U0 = state["U0"].detach().requires_grad_()
    U0.grad = None
    UT = FvRunFunction.apply(U0, s, case["steps"], state["dt"], case["every"])
    kinetic_energy(UT, state["grid"]).backward()
    return {"U": UT.detach(), "g": U0.grad}


def work(case):
    kind = case["kind"]
    if kind == "surrogate":
        sizes = [case["features"], 128, 64, 32, 1]
        macs = sum(a * b for a, b in zip(sizes[:-1], sizes[1:]))
        npar = macs + sum(sizes[1:])
        return {"bytes": 8.0 * (2 * npar + (case["train"] + case["candidates"]) * (case["features"] + 1))
                + 4.0 * case["train"] * case["epochs"],
                "flops": 6.0 * macs * case["train"] * case["epochs"] + 2.0 * macs * case["candidates"]}
    if kind == "batch":
        cells = sum(n * n for n, _ in I.batched_sod(case["count"], case["sizes_seed"], case["nmin"], case["nmax"]))
        return {"bytes": 2.0 * 32 * cells, "flops": 3.0 * FLOP_CELL_STAGE[2] * cells * case["steps"]}
    d = case["dim"]
    cells = case["nx"] * case["ny"] * case["nz"]
    state = 8.0 * (d + 2) * cells
    one = FLOP_CELL_STAGE[d] * cells
    if kind == "residual":
        return {"bytes": 2 * state, "flops": one}
    if kind in ("run", "host_run"):
        return {"bytes": (3 if case.get("source") else 2) * state, "flops": 3 * one * case["steps"]}
    if kind == "vjp":  # the reverse of an evaluation costs about twice the evaluation that it repeats
        return {"bytes": 3 * state, "flops": 3 * one}
    if kind == "step_vjp":
        return {"bytes": 3 * state, "flops": (2 + 9) * one}
    return {"bytes": 3 * state, "flops": (3 + 3 + 9) * one * case["steps"]}


# ----------------------------------------------------------------------------- the same in plain 64-bit torch

def _shift(U, axis, k, periodic):
    """U at index i + k along axis, with the ghost cells of the boundary."""
    n = U.shape[axis]
    i = torch.arange(n, device=U.device) + k
    i = i % n if periodic else i.clamp(0, n - 1)
    return U.index_select(axis, i)


def _limited(a, b, limiter):
    if limiter == "none":
        return a
    same = a * b > 0.0
    zero = torch.zeros_like(a)
    if limiter == "vanleer":
        return torch.where(same, 2.0 * a * b / torch.where(same, a + b, torch.ones_like(a)), zero)
    return torch.where(same, torch.where(a.abs() < b.abs(), a, b), zero)


def _roe(QL, QR, ax, dim, efix=0.1):
    g1 = GAMMA - 1.0

    def prim(Q):
        u = [Q[1 + d] / Q[0] for d in range(dim)]
        p = g1 * (Q[-1] - 0.5 * sum(Q[1 + d] * u[d] for d in range(dim)))
        return u, p, (Q[-1] + p) / Q[0]

    uL, pL, HL = prim(QL)
    uR, pR, HR = prim(QR)
    sL, sR = QL[0].sqrt(), QR[0].sqrt()
    inv = 1.0 / (sL + sR)
    u = [(sL * a + sR * b) * inv for a, b in zip(uL, uR)]
    H = (sL * HL + sR * HR) * inv
    q2 = sum(v * v for v in u)
    c = (g1 * (H - 0.5 * q2)).sqrt()
    rho = sL * sR
    du = [b - a for a, b in zip(uL, uR)]
    dp = pR - pL
    a1 = (dp - rho * c * du[ax]) / (2.0 * c * c)
    a2 = QR[0] - QL[0] - dp / (c * c)
    a3 = (dp + rho * c * du[ax]) / (2.0 * c * c)
    delta = efix * c

    def fixed(lam):
        return torch.where(lam.abs() < delta, (lam * lam + delta * delta) / (2.0 * delta), lam.abs())

    w1, w2, w3 = fixed(u[ax] - c) * a1, u[ax].abs() * a2, fixed(u[ax] + c) * a3
    sh = [u[ax].abs() * rho * d for d in du]
    F = [0.5 * (QL[1 + ax] + QR[1 + ax]) - 0.5 * (w1 + w2 + w3)]
    for d in range(dim):
        f = 0.5 * (QL[1 + d] * uL[ax] + QR[1 + d] * uR[ax])
        if d == ax:
            f = f + 0.5 * (pL + pR) - 0.5 * (w1 * (u[d] - c) + w2 * u[d] + w3 * (u[d] + c))
        else:
            f = f - 0.5 * ((w1 + w2 + w3) * u[d] + sh[d])
        F.append(f)
    FE = 0.5 * ((QL[-1] + pL) * uL[ax] + (QR[-1] + pR) * uR[ax])
    FE = FE - 0.5 * (w1 * (H - u[ax] * c) + w2 * 0.5 * q2 + w3 * (H + u[ax] * c))
    for d in range(dim):
        if d != ax:
            FE = FE - 0.5 * sh[d] * u[d]
    F.append(FE)
    return F


def _tendency(U, g, limiter="minmod", recon="conserved", S=None, area=False):
    """dU/dt, or with area the residual (face areas included)."""
    dim = g.dim
    h = g.spacing
    g1 = GAMMA - 1.0
    out = torch.zeros_like(U) if S is None else S.clone()
    W = U
    if recon == "primitive":
        u = [U[1 + d] / U[0] for d in range(dim)]
        W = torch.stack([U[0]] + u + [g1 * (U[-1] - 0.5 * U[0] * sum(v * v for v in u))])
    for ax in range(dim):
        axis = dim - ax
        per = g.bc[ax][0] == I.BC_PERIODIC
        n = g.n[ax]
        # faces 0..n along the axis: face f between cells f - 1 and f
        ids = torch.arange(-2, n + 2, device=U.device)
        ids = ids % n if per else ids.clamp(0, n - 1)
        P = W.index_select(axis, ids)
        q = [P.narrow(axis, k, n + 1) for k in range(4)]
        dm, d0, dp = q[1] - q[0], q[2] - q[1], q[3] - q[2]
        QL, QR = q[1] + 0.5 * _limited(dm, d0, limiter), q[2] - 0.5 * _limited(dp, d0, limiter)
        if limiter == "minmod":  # on ties the second argument of the ordered pair
            QL, QR = q[1] + 0.5 * _limited(dm, d0, limiter), q[2] - 0.5 * _limited(d0, dp, limiter)
        if recon == "primitive":
            def cons(w):
                return [w[0]] + [w[0] * w[1 + d] for d in range(dim)] + \
                    [w[-1] / g1 + 0.5 * w[0] * sum(w[1 + d] ** 2 for d in range(dim))]
            QL, QR = cons(QL), cons(QR)
        F = torch.stack(_roe(list(QL), list(QR), ax, dim))
        del q, dm, d0, dp, QL, QR, P
        out = out - (F.narrow(axis, 1, n) - F.narrow(axis, 0, n)) / h[ax]
        del F
    if area:
        out = -out * math.prod(h[:dim])
    return out


def _cfl_step(U, g):
    u = [U[1 + d] / U[0] for d in range(g.dim)]
    p = (GAMMA - 1.0) * (U[-1] - 0.5 * U[0] * sum(v * v for v in u))
    c = (GAMMA * p / U[0]).sqrt()
    return 0.5 / float(sum((u[d].abs() + c) / g.spacing[d] for d in range(g.dim)).max())


def _rk3(U, dt, f):
    U1 = U + dt * f(U)
    U2 = 0.75 * U + 0.25 * (U1 + dt * f(U1))
    return U / 3.0 + (2.0 / 3.0) * (U2 + dt * f(U2))


def exact(case, seed):
    kind = case["kind"]
    if kind == "surrogate":
        return _exact_surrogate(case, seed)
    if kind == "batch":
        grids, states = _batch_states(case, seed)
        parts, at = [], 0
        for g, U in zip(grids, states):
            for _ in range(case["steps"]):
                U = _rk3(U, _cfl_step(U, g), lambda V: _tendency(V, g))
            pad = -at % 32  # blocks start on 256-byte boundaries
            parts += [torch.zeros(pad, dtype=torch.float64, device="cuda"), U.reshape(-1)]
            at += pad + U.numel()
        parts.append(torch.zeros(-at % 32, dtype=torch.float64, device="cuda"))
        return {"U": torch.cat(parts)}
    g = _grid(case)
    U = _state(case, g, seed)
    opt = dict(limiter=case.get("limiter", "minmod"), recon=case.get("recon", "conserved"))
    if kind == "residual":
        R = _tendency(U, g, area=True, **opt)
        return {"R": R, "norms": (R * R).reshape(g.nvar, -1).sum(dim=1)}
    if kind in ("run", "host_run"):
        S = _source(g, seed) if case.get("source") else None
        for _ in range(case["steps"]):
            U = _rk3(U, _cfl_step(U, g), lambda V: _tendency(V, g, S=S, **opt))
        return {"U": U.cpu().numpy() if kind == "host_run" else U}
    dt = _cfl_step(U, g)
    if kind in ("vjp", "step_vjp"):
        lam = _cotangent(g, seed)
        V = U.requires_grad_()
        y = _tendency(V, g, area=True) if kind == "vjp" else _rk3(V, dt, lambda W: _tendency(W, g))
        return {"g": torch.autograd.grad(y, V, lam)[0]}
    states = [U]
    with torch.no_grad():
        for _ in range(case["steps"]):
            states.append(_rk3(states[-1], dt, lambda W: _tendency(W, g)))
    UT = states.pop().requires_grad_()
    lam = torch.autograd.grad(kinetic_energy_plain(UT, g), UT)[0]
    while states:
        V = states.pop().requires_grad_()
        lam = torch.autograd.grad(_rk3(V, dt, lambda W: _tendency(W, g)), V, lam)[0]
    return {"U": UT.detach(), "g": lam}


def kinetic_energy_plain(U, g):
    return (0.5 * sum(U[1 + d] ** 2 for d in range(g.dim)) / U[0]).sum() * math.prod(g.spacing[:g.dim])


def _exact_surrogate(case, seed):
    sizes, flat, X, y, order, C = _surrogate_data(case, seed)
    order = order.long()
    views, k = [], 0
    for fi, fo in zip(sizes[:-1], sizes[1:]):
        views.append((flat[k:k + fi * fo].view(fi, fo), flat[k + fi * fo:k + fi * fo + fo]))
        k += fi * fo + fo
    m, v, t, losses = torch.zeros_like(flat), torch.zeros_like(flat), 0, []
    h = fv.mlp_hyper()

    def forward(A):
        acts = [A]
        for l, (W, b) in enumerate(views):
            Z = acts[-1] @ W + b
            acts.append(Z.clamp_min(0.0) if l < len(views) - 1 else Z)
        return acts

    for ep in range(case["epochs"]):
        total = torch.zeros((), dtype=torch.float64, device="cuda")
        for s0 in range(0, case["train"], h.batch):
            idx = order[ep, s0:s0 + h.batch]
            acts = forward(X[idx])
            delta = acts[-1] - y[idx][:, None]
            total = total + 0.5 * (delta * delta).sum() + 0.5 * h.alpha * sum((W * W).sum() for W, _ in views)
            grads = []
            for l in range(len(views) - 1, -1, -1):
                W = views[l][0]
                grads = [((acts[l].T @ delta + h.alpha * W) / len(idx)).reshape(-1), delta.mean(dim=0)] + grads
                if l > 0:
                    delta = (delta @ W.T) * (acts[l] > 0.0)
            gr = torch.cat(grads)
            t += 1
            m = h.beta1 * m + (1.0 - h.beta1) * gr
            v = h.beta2 * v + (1.0 - h.beta2) * gr * gr
            flat -= h.lr * math.sqrt(1.0 - h.beta2 ** t) / (1.0 - h.beta1 ** t) * m / (v.sqrt() + h.eps)
        losses.append(float(total) / case["train"])
    return {"params": flat, "scores": forward(C)[-1][:, 0], "losses": np.array(losses)}
