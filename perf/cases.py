"""The work this framework does for its users, as cases that can be timed and compared.

A case is a dict of plain values; `prepare` makes what a user's program holds before
the call, `run` is one pass through the public entry points of
``paper_1302_3663_gb300.bfibm``. Sizes and settings are those of the workloads in
``paper_1302_3663_gb300/workloads.py``, ``bench.py`` and the tests:

* whole time steps (what every user runs): 2D and 3D, plain FP64 with fixed V-cycles,
  the open duct, mixed precision to a tolerance, and batches of uneven ducts;
* the two multigrid solves and the FP64 smoothers alone, on seeded coefficients and
  right-hand sides, where the answer is known in closed form by a linear system.
"""
import math

import numpy as np
import torch

from paper_1302_3663_gb300 import bfibm, workloads as W

# the benchmark's solver (bench.py): both solves to max |div u| <= 1e-10
TOL = {"vc_visc": 0, "vc_p": 0, "rtol": 1e-11, "max_cycles": 100, "gamma_coarse": 0.8, "nu1": 2,
       "nu2": 2, "inner_cycles": 2, "krylov": 1, "div_tol": 1e-10}


def listed():
    return [
        # the 2D biofilm workload: 64x32, 150 nodes, 20 steps of 3 V-cycles per solve. The
        # smallest simulation: launches and latency count, not arithmetic.
        dict(name="step2d_64x32", kind="step2d", n=64, steps=20),
        # one resolution of the 2D refinement study (h = 1/256), the same 150 nodes
        dict(name="step2d_256x128", kind="step2d", n=256, steps=5),
        # the 64^3 square duct in plain FP64, 2,000 nodes, 3 V-cycles per solve
        dict(name="step3d_fp64_64", kind="step3d", e=64, length=64, nodes=2000, open=False,
             steps=4),
        # the open duct (inflow, outflow) of 64x64x128 cells in FP64
        dict(name="open3d_fp64_64", kind="step3d", e=64, length=128, nodes=2000, open=True,
             steps=2),
        # the smallest request of the serving stream, mixed precision to a tolerance
        dict(name="mixed_48", kind="mixed", e=48, ey=48, nodes=500),
        # a request whose coarse grids do not halve far: 144 / 16 = 9
        dict(name="mixed_144", kind="mixed", e=144, ey=144, nodes=50000),
        # the headline: the 128x128x256 duct with 20,000 nodes
        dict(name="mixed_128", kind="mixed", e=128, ey=128, nodes=20000),
        # the batched sweep: uneven ducts of edges 32..96 in lock step
        dict(name="batch_persistent_12", kind="batch", members=12, persistent=True),
        # a handful of such simulations as the service runs them by default: each on its stream
        dict(name="batch_replay_6", kind="batch", members=6, persistent=False),
        # the viscous solve alone (flexible CG around FP32 V-cycles), viscosity ratio 1e3
        dict(name="solve_visc_96", kind="solve_visc", nx=96, ny=96, nz=192, mixed=True),
        # the pressure solve alone at the largest request size
        dict(name="solve_p_160", kind="solve_p", nx=160, ny=160, nz=320, mixed=True),
        # the FP64 smoothers alone on a ragged grid
        dict(name="sweeps_fp64_ragged", kind="sweeps", nx=101, ny=75, nz=130, sweeps=3),
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step2d", "step3d", "open3d", "mixed", "batch", "solve_visc", "solve_p",
                       "sweeps"])
    if kind == "step2d":
        # widths with at least two halvings, odd quotients among them
        return dict(kind="step2d", n=4 * _logint(rng, 8, 64), steps=rng.randint(1, 20))
    if kind in ("step3d", "open3d"):
        e = 8 * rng.randint(4, 8)
        return dict(kind="step3d", e=e, length=rng.choice([1, 2]) * e,
                    nodes=_logint(rng, 200, 2000), open=kind == "open3d", steps=rng.randint(1, 4))
    if kind == "mixed":
        # edges of the serving stream's range, the cross section square or flat
        e = 16 * rng.randint(3, 8)
        return dict(kind="mixed", e=e, ey=max(48, e - 16 * rng.randint(0, 2)),
                    nodes=_logint(rng, 500, 50000))
    if kind == "batch":
        return dict(kind="batch", members=rng.randint(2, 12), persistent=rng.random() < 0.5)
    if kind in ("solve_visc", "solve_p"):
        return dict(kind=kind, nx=8 * rng.randint(4, 16), ny=8 * rng.randint(4, 16),
                    nz=16 * rng.randint(2, 16), mixed=rng.random() < 0.75)
    return dict(kind="sweeps", nx=_logint(rng, 9, 128), ny=_logint(rng, 9, 128),
                nz=2 * _logint(rng, 4, 64), sweeps=rng.randint(1, 3))


# --------------------------------------------------------------------------- steps
def _mixed_instance(e, ey, nodes, seed):
    """A request of the serving stream: an e x ey x 2e duct with three Gaussian mounds."""
    rng = np.random.Generator(np.random.PCG64(seed))
    h, r, sig = 1.0 / e, 0.005, 0.05
    counts = [nodes // 3 + (1 if q < nodes % 3 else 0) for q in range(3)]
    X = W.gaussian_mounds(rng, counts, [(0.5, 0.0, 0.5), (0.5, 0.0, 1.0), (0.5, 0.0, 1.5)], sig,
                          (0, 0, 0), (1, ey * h, 2))
    vol = 3 * 2.0 / 3.0 * math.pi * (2.0 * sig) ** 3
    prm = W.base_params(3, (e, ey, 2 * e), (0, 0, 1), 2, h, rho_ratio=2.0, mu_ratio=1e3, omega=r,
                        omega_mu=r, d0_vol=vol / nodes, **dict(TOL, precision=1))
    return _with_springs(prm, X, r, rng)


def _with_springs(prm, X, r, rng):
    ab, rest = W.springs_within(X, 2.5 * r)
    K = np.exp(rng.uniform(math.log(0.1), math.log(10.0), size=ab.shape[0]))
    return dict(params=prm, X=X, ab=ab, rest=rest, K=K, brk=np.full(ab.shape[0], 0.3))


def _sweep_instance(i, seed):
    """Duct i of the batched sweep: e x e x 2e, edges 32..96 in turn, 500-8,000 nodes uniform in
    the hemispherical mound, density ratio in [1, 2], viscosity ratio in [10, 1000]."""
    rng = np.random.Generator(np.random.PCG64([seed, i]))
    e, m, r, R = (64, 32, 96, 48)[i % 4], 500 + 7500 * (i * 5 % 12) // 11, 0.008, 0.15
    c = rng.normal(size=(m, 3))
    X = c * (R * rng.uniform(size=(m, 1)) ** (1 / 3) / np.linalg.norm(c, axis=1, keepdims=True))
    X[:, 1] = np.abs(X[:, 1])
    X += (0.5, 0.0, 1.0)
    prm = W.base_params(3, (e, e, 2 * e), (0, 0, 1), 2, 1.0 / e, rho_ratio=rng.uniform(1.0, 2.0),
                        mu_ratio=math.exp(rng.uniform(math.log(10.0), math.log(1e3))), omega=r,
                        omega_mu=r, d0_vol=2.0 / 3.0 * math.pi * R ** 3 / m,
                        **dict(TOL, precision=1))
    return _with_springs(prm, X, r, rng)


def _fp64_instance(case, seed):
    """The hemispherical mound of the 64^3 duct workload on an e x e x length duct."""
    rng = np.random.Generator(np.random.PCG64(seed))
    e, m, r, R = case["e"], case["nodes"], 0.008, 0.15
    X, _ = W.dart_throw(rng, m, 3, (0.5, 0.0, 0.5), R, 2 * r, attempts_per_node=6)
    h = 1.0 / e
    prm = W.base_params(3, (e, e, case["length"]), (0, 0, 0 if case["open"] else 1), 2, h,
                        rho_ratio=1.5, mu_ratio=1e3, omega=r, omega_mu=r,
                        d0_vol=2.0 / 3.0 * math.pi * R ** 3 / m, open_flow=int(case["open"]))
    return _with_springs(prm, X, r, rng)


def _read(ctx):
    """What a run is read for: velocity and pressure (on the device) and the nodes."""
    out = {}
    for name, which, comp in [("u%d" % d, "u", d) for d in range(ctx.dim)] + [("p", "p", 0)]:
        t = torch.empty(ctx.shape(), dtype=torch.float64, device="cuda")
        ctx.get_field_dev(which, t.data_ptr(), comp)
        out[name] = t
    out["X"] = ctx.get_nodes()
    return out


# ----------------------------------------------------- seeded operators for the solves
def _bumps(nz, ny, nx, seed, device):
    """Smooth-edged blobs on the y = 0 wall with cell-scale grain, in [0, 1], on one grid of
    points per staggering: drawn on the whole index grid, so every staggering has its own."""
    g = torch.Generator(device="cpu").manual_seed(seed)
    grain = torch.rand((nz, ny, nx), generator=g, dtype=torch.float64).to(device)
    z = torch.arange(nz, dtype=torch.float64, device=device).view(-1, 1, 1) / nz
    y = torch.arange(ny, dtype=torch.float64, device=device).view(1, -1, 1) / ny
    x = torch.arange(nx, dtype=torch.float64, device=device).view(1, 1, -1) / nx
    r2 = (x - 0.5) ** 2 + y ** 2 + 0.25 * torch.sin(math.pi * 3 * z) ** 2
    return ((0.06 - r2) * 40 + grain - 0.5).clamp(0, 1)


def _system(case, seed):
    """Coefficients, start and right-hand sides of a solve on [0,1]-wide ducts (walls in x and
    y, periodic z), in the dense field layout (nz, ny + 1, nx + 1), all from the seed."""
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    dev = "cuda"
    sh = (nz, ny + 1, nx + 1)
    h = 1.0 / max(nx, ny)
    S = {"n": (nx, ny, nz), "h": h, "dt": 0.1 * h}
    S["rho"] = [1.0 + _bumps(*sh, seed * 16 + d, dev) for d in range(3)]
    mu = [0.01 * 1e3 ** _bumps(*sh, seed * 16 + 3 + e, dev) for e in range(4)]
    S["muc"], S["mue"] = mu[0], mu[1:]
    g = torch.Generator(device="cpu").manual_seed(seed * 16 + 9)

    def rand():
        return torch.randn(sh, generator=g, dtype=torch.float64).to(dev)

    y = (torch.arange(ny + 1, dtype=torch.float64, device=dev).view(1, -1, 1) + 0.5) / ny
    x = (torch.arange(nx + 1, dtype=torch.float64, device=dev).view(1, 1, -1) + 0.5) / nx
    flow = (16 * x * (1 - x) * y * (1 - y)).expand(sh)
    S["u0"] = [0.05 * rand() + (flow if d == 2 else 0.0) for d in range(3)]
    S["f"] = [S["rho"][d] / S["dt"] * (S["u0"][d] + 0.05 * rand()) for d in range(3)]
    for d in range(3):
        m = _faces(S["n"], d, dev)
        S["u0"][d] = torch.where(m, S["u0"][d], 0.0)
        S["f"][d] = torch.where(m, S["f"][d], 0.0)
    b = rand()
    c = _cells(S["n"], dev)
    b = torch.where(c, b, 0.0)
    S["b"] = torch.where(c, (b - b.sum() / c.sum()) / (S["dt"] * h), 0.0)
    S["p0"] = torch.where(c, 0.01 * rand(), 0.0)
    return S


def _cells(n, dev):
    m = torch.zeros((n[2], n[1] + 1, n[0] + 1), dtype=torch.bool, device=dev)
    m[:, :n[1], :n[0]] = True
    return m


def _faces(n, d, dev):
    """Unknown faces of component d."""
    m = _cells(n, dev)
    if d == 0:
        m[:, :, 0] = False
    if d == 1:
        m[:, 0, :] = False
    return m


def _prm(case):
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    h = 1.0 / max(nx, ny)
    prm = W.base_params(3, (nx, ny, nz), (0, 0, 1), 2, h, rho_ratio=2.0, mu_ratio=1e3,
                        omega=2 * h, omega_mu=2 * h, d0_vol=h ** 3)
    if case["kind"] != "sweeps":
        prm.update(TOL, precision=int(case["mixed"]))
        prm["div_tol"] = 0.0
    return prm


def _load_system(case, seed):
    S = _system(case, seed)
    ctx = bfibm.Context(_prm(case))
    for d in range(3):
        ctx.set_field_dev("rho", S["rho"][d].data_ptr(), d)
        ctx.set_field_dev("mue", S["mue"][d].data_ptr(), d)
    ctx.set_field_dev("muc", S["muc"].data_ptr())
    ctx.build_coefficients()
    if case["kind"] != "solve_p":
        for d in range(3):
            ctx.set_field_dev("urhs", S["f"][d].data_ptr(), d)
    if case["kind"] != "solve_visc":
        ctx.set_field_dev("prhs", S["b"].data_ptr())
    return dict(ctx=ctx, u0=S["u0"], p0=S["p0"], kind=case["kind"], sweeps=case.get("sweeps", 0))


# ------------------------------------------------------------------- the entry points
def prepare(case, seed):
    kind = case["kind"]
    if kind in ("step2d", "step3d", "mixed"):
        if kind == "step2d":
            inst = W.mound_2d(case["n"], rho_ratio=1.5, mu_ratio=100.0, omega=0.01, seed=seed)
        elif kind == "step3d":
            inst = _fp64_instance(case, seed)
        else:
            inst = _mixed_instance(case["e"], case["ey"], case["nodes"], seed)
        ctx = bfibm.load_instance(inst)
        ctx.refresh()
        return dict(kind=kind, ctx=ctx, steps=case.get("steps", 1))
    if kind == "batch":
        batch = bfibm.Batch(persistent=case["persistent"], tune=False)
        ctxs = []
        for i in range(case["members"]):
            ctx = bfibm.load_instance(_sweep_instance(i, seed))
            ctx.set_option(bfibm.OPT_STATS, 0)
            batch.add(ctx)
            ctxs.append(ctx)
        return dict(kind=kind, batch=batch, ctxs=ctxs)
    return _load_system(case, seed)


def run(state):
    kind = state["kind"]
    if kind == "batch":
        state["batch"].step()
        state["batch"].wait()
        return [_read(c) for c in state["ctxs"]]
    ctx = state["ctx"]
    if kind in ("step2d", "step3d", "mixed"):
        ctx.step(state["steps"])
        return _read(ctx)
    visc, pres = kind != "solve_p", kind != "solve_visc"
    if visc:
        for d in range(3):
            ctx.set_field_dev("ut", state["u0"][d].data_ptr(), d)
    if pres:
        ctx.set_field_dev("p", state["p0"].data_ptr())
    if kind == "solve_visc":
        ctx.solve_viscous(0)
    elif kind == "solve_p":
        ctx.solve_pressure(0)
    else:
        ctx.smooth_viscous(0, state["sweeps"], sync=False)
        ctx.smooth_pressure(0, state["sweeps"], sync=False)
    out = {}
    for name, which, comp in ([("ut%d" % d, "ut", d) for d in range(3)] if visc else []) + \
            ([("p", "p", 0)] if pres else []):
        t = torch.empty(ctx.shape(), dtype=torch.float64, device="cuda")
        ctx.get_field_dev(which, t.data_ptr(), comp)
        out[name] = t
    return out


def work(case):
    """State in and state out, once per step or solve; the arithmetic of one pass of the two
    operators over the grid (what any solver applies at least once)."""
    kind = case["kind"]
    if kind == "step2d":
        cells, steps, per, ops = case["n"] * case["n"] // 2, case["steps"], 8 * 6, 60
    elif kind == "step3d":
        cells, steps, per, ops = case["e"] ** 2 * case["length"], case["steps"], 8 * 8, 120
    elif kind == "mixed":
        cells, steps, per, ops = case["e"] * case["ey"] * 2 * case["e"], 1, 8 * 8, 120
    elif kind == "batch":
        cells = sum(2 * (64, 32, 96, 48)[i % 4] ** 3 for i in range(case["members"]))
        steps, per, ops = 1, 8 * 8, 120
    else:
        cells, steps = case["nx"] * case["ny"] * case["nz"], max(1, case.get("sweeps", 1))
        # viscous: u in and out, f, m (or rho), mu on centres and edges; pressure: p, b, beta
        per = {"solve_visc": 8 * 16, "solve_p": 8 * 6, "sweeps": 8 * 22}[kind]
        ops = {"solve_visc": 90, "solve_p": 20, "sweeps": 110}[kind]
    return {"bytes": float(cells * steps * per), "flops": float(cells * steps * ops)}


# ------------------------------------------------------------------------ in 64 bits
def _roll_m(f, axis):   # value at index - 1 (zero beyond the lower wall, periodic in z)
    if axis == 2:
        return torch.roll(f, 1, 0)
    out = torch.zeros_like(f)
    if axis == 1:
        out[:, 1:, :] = f[:, :-1, :]
    else:
        out[:, :, 1:] = f[:, :, :-1]
    return out


def _roll_p(f, axis):
    if axis == 2:
        return torch.roll(f, -1, 0)
    out = torch.zeros_like(f)
    if axis == 1:
        out[:, :-1, :] = f[:, 1:, :]
    else:
        out[:, :, :-1] = f[:, :, 1:]
    return out


def _at(n, axis, i, dev):   # mask of the index plane i along an axis
    m = torch.zeros((n[2], n[1] + 1, n[0] + 1), dtype=torch.bool, device=dev)
    if axis == 0:
        m[:, :, i] = True
    elif axis == 1:
        m[:, i, :] = True
    else:
        m[i] = True
    return m


_EDGE = {(0, 1): 0, (0, 2): 1, (1, 2): 2}


def _visc(S, u, d, ir):
    """(A u)_d = m_d u_d - (1/Re) [div (mu (grad u + grad u^T))]_d on the unknown faces."""
    n, dev = S["n"], u[0].device
    tau = 2 * S["muc"] * (_roll_p(u[d], d) - u[d])
    V = tau - _roll_m(tau, d)
    for e in range(3):
        if e == d:
            continue
        mu = S["mue"][_EDGE[tuple(sorted((d, e)))]]
        below = _roll_m(u[d], e)
        if e < 2:   # mirror ghosts beyond the walls: at the edge 0 and at the edge n
            below = torch.where(_at(n, e, 0, dev), -u[d], below)
            here = torch.where(_at(n, e, n[e], dev), -below, u[d])
        else:
            here = u[d]
        t = mu * ((here - below) + (u[e] - _roll_m(u[e], d)))
        V = V + _roll_p(t, e) - t
    return torch.where(_faces(n, d, dev), S["rho"][d] / S["dt"] * u[d] - ir * V, 0.0)


def _visc_diag(S, d, ir):
    n, dev = S["n"], S["muc"].device
    g = 2 * (S["muc"] + _roll_m(S["muc"], d))
    for e in range(3):
        if e == d:
            continue
        mu = S["mue"][_EDGE[tuple(sorted((d, e)))]]
        if e < 2:
            mu = mu * torch.where(_at(n, e, 0, dev) | _at(n, e, n[e], dev), 2.0, 1.0)
        g = g + mu + _roll_p(mu, e)
    return S["rho"][d] / S["dt"] + ir * g


def _beta(S):
    """1/rho on the faces fluxes cross (0 on the walls)."""
    return [torch.where(_faces(S["n"], a, S["b"].device), 1.0 / S["rho"][a], 0.0)
            for a in range(3)]


def _pres(S, beta, p):
    r = torch.zeros_like(p)
    for a in range(3):
        fl = beta[a] * (p - _roll_m(p, a))
        r = r + _roll_p(fl, a) - fl
    return torch.where(_cells(S["n"], p.device), r / S["h"] ** 2, 0.0)


def _pres_diag(S, beta):
    g = sum(b + _roll_p(b, a) for a, b in enumerate(beta))
    return torch.where(_cells(S["n"], S["b"].device), g / S["h"] ** 2, 1.0)


def _cg(apply, b, x, inv_diag, tol=1e-14, most=6000):
    def dot(a, c):
        return sum((p * q).sum() for p, q in zip(a, c))

    r = [f - a for f, a in zip(b, apply(x))]
    z = [q * i for q, i in zip(r, inv_diag)]
    p = list(z)
    rz, stop = dot(r, z), tol * math.sqrt(float(dot(b, b)))
    for it in range(most):
        q = apply(p)
        alpha = rz / dot(p, q)
        x = [a + alpha * c for a, c in zip(x, p)]
        r = [a - alpha * c for a, c in zip(r, q)]
        if it % 20 == 19 and math.sqrt(float(dot(r, r))) < stop:
            break
        z = [a * i for a, i in zip(r, inv_diag)]
        new = dot(r, z)
        p = [a + (new / rz) * c for a, c in zip(z, p)]
        rz = new
    return x


def exact(case, seed):
    """The solves' answers (a linear system, by conjugate gradients to rounding) and the
    smoothers' (point by point). A whole time step has no value but the method's own."""
    kind = case["kind"]
    if kind not in ("solve_visc", "solve_p", "sweeps"):
        return None
    S = _system(case, seed)
    ir, dev = 1.0 / S["h"] ** 2, S["b"].device
    beta = _beta(S)
    if kind == "solve_visc":
        inv = [1.0 / _visc_diag(S, d, ir) for d in range(3)]
        u = _cg(lambda v: [_visc(S, v, d, ir) for d in range(3)], S["f"], S["u0"], inv)
        return {"ut%d" % d: u[d] for d in range(3)}
    if kind == "solve_p":
        inv = 1.0 / _pres_diag(S, beta)
        p = _cg(lambda v: [-_pres(S, beta, v[0])], [-S["b"]], [S["p0"]], [inv])[0]
        c = _cells(S["n"], dev)
        return {"p": torch.where(c, p - p.sum() / c.sum(), 0.0)}
    n = S["n"]
    parity = (torch.arange(n[2], device=dev).view(-1, 1, 1) +
              torch.arange(n[1] + 1, device=dev).view(1, -1, 1) +
              torch.arange(n[0] + 1, device=dev).view(1, 1, -1)) % 2
    u, p = list(S["u0"]), S["p0"]
    vd = [_visc_diag(S, d, ir) for d in range(3)]
    pd = -_pres_diag(S, beta)
    cells = _cells(n, dev)
    for _ in range(case["sweeps"]):
        for d in range(3):
            for colour in (0, 1):
                new = u[d] + (S["f"][d] - _visc(S, u, d, ir)) / vd[d]
                u[d] = torch.where(_faces(n, d, dev) & (parity == colour), new, u[d])
        for colour in (0, 1):
            new = p + (S["b"] - _pres(S, beta, p)) / pd
            p = torch.where(cells & (parity == colour), new, p)
    out = {"ut%d" % d: u[d] for d in range(3)}
    out["p"] = p
    return out
