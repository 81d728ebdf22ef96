"""The work that programs have this library do, as cases to be timed and compared.

Five kinds of call, each through the package's public entry points:

* ``step``      one implicit (or explicit) time step of a flow: the whole call
                of a time loop (ROW, ESDIRK, BDF2, SSPRK3);
* ``operator``  ``fr_residual`` and ``fr_jv``: R(U) and the finite-difference
                product A z that an outer solver asks for;
* ``blocks``    ``ejacobi_factor`` and ``ejacobi_apply``: the element-Jacobi
                preconditioner formed, inverted and applied once;
* ``batch``     one ROW step of several independent instances;
* ``train`` / ``infer``  the per-element network of the learned initial guess:
                one FP32 training step, one BF16 inference.

Flows: ``vortex`` (2D Euler, the isentropic vortex on a periodic square),
``channel`` (2D Navier-Stokes between walls, mesh clustered towards them),
``tgv`` (3D Navier-Stokes, the Taylor-Green vortex on a periodic cube).
"""
import math

import numpy as np
import torch

GAMMA = 1.4
SHIFT = 1.0 / (0.435866521508459 * 0.05)   # 1 / (gamma dt) of a ROW3 step of 0.05


# ------------------------------------------------------------------ cases --

def listed():
    return [
        # the small configuration: a second-order ROW step of the 20 x 20 vortex; every
        # launch is microseconds long, so latency and launches count
        dict(name="step-row2-vortex-20x20-p2", kind="step", flow="vortex", scheme="row2", nx=20, ny=20, p=2,
             precision=0, riemann=0, jv=0, dt=0.05, tol=1e-8),
        # the main configuration: one ROW3 step of the 160 x 160 vortex at CFL 13.6
        dict(name="step-row3-vortex-160x160-p3", kind="step", flow="vortex", scheme="row3", nx=160, ny=160, p=3,
             precision=0, riemann=0, jv=0, dt=0.05, tol=1e-6),
        # pseudo-transient continuation with many loose inner solves and re-inverted BF16
        # blocks: an ESDIRK3 step of the wall-bounded channel
        dict(name="step-esdirk3-channel-64x64-p3", kind="step", flow="channel", scheme="esdirk3", nx=64, ny=64, p=3,
             precision=2, riemann=0, jv=0, dt=1e-3, tol=0.1),
        # R(U) and A z alone at the smallest size: the smallest calls a program makes
        dict(name="operator-vortex-20x20-p2", kind="operator", flow="vortex", nx=20, ny=20, p=2, riemann=0, jv=0,
             stretch=0.0),
        # the same at a large size, stretched mesh
        dict(name="operator-vortex-512x512-p3", kind="operator", flow="vortex", nx=512, ny=512, p=3, riemann=0, jv=0,
             stretch=0.3),
        # the viscous (BR2) operator on the channel mesh
        dict(name="operator-channel-256x128-p3", kind="operator", flow="channel", nx=256, ny=128, p=3),
        # the 3D operator of the Taylor-Green study
        dict(name="operator-tgv-32x32x32-p3", kind="operator", flow="tgv", nx=32, ny=32, nz=32, p=3, jv=0),
        # the FP64 element blocks of the main configuration: formed, inverted, applied
        dict(name="blocks-vortex-160x160-p3", kind="blocks", flow="vortex", nx=160, ny=160, p=3, precision=0,
             riemann=0),
        # the 320-row blocks of the 3D study: FP32 columns, stored in BF16
        dict(name="blocks-tgv-16x16x16-p3", kind="blocks", flow="tgv", nx=16, ny=16, nz=16, p=3, precision=2,
             columns=1),
        # independent instances of uneven size and degree stepped together
        dict(name="batch-8-row4", kind="batch", count=8, smallest=32, largest=96, precision=2, dt=0.05, tol=1e-6),
        # one optimiser step of the guess network on a minibatch of captured stage solves
        dict(name="train-8192-nb100", kind="train", rows=8192, nb=100),
        # the guess for every element of a 384 x 192 mesh at p = 4
        dict(name="infer-73728-nb100", kind="infer", rows=73728, nb=100),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    pick = rng.choice(["step", "step", "step", "operator", "operator", "operator", "blocks", "blocks", "batch", "net"])
    if pick == "net":
        nb = rng.choice([36, 64, 100])
        if rng.random() < 0.5:
            return dict(kind="train", rows=_log(rng, 256, 8192), nb=nb)
        return dict(kind="infer", rows=_log(rng, 1000, 73728), nb=nb)
    if pick == "batch":
        return dict(kind="batch", count=rng.randint(2, 8), smallest=rng.randint(12, 32), largest=rng.randint(40, 96),
                    precision=rng.choice([0, 2]), dt=round(rng.uniform(0.02, 0.06), 4), tol=1e-6)
    flow = rng.choice(["vortex", "vortex", "channel", "tgv"])
    if pick == "operator":
        if flow == "vortex":
            return dict(kind="operator", flow=flow, nx=_log(rng, 7, 400), ny=_log(rng, 7, 400),
                        p=rng.choice([2, 3, 3, 4, 5, 6]), riemann=rng.choice([0, 0, 1]), jv=rng.choice([0, 0, 0, 1]),
                        stretch=rng.choice([0.0, 0.3]))
        if flow == "channel":
            return dict(kind="operator", flow=flow, nx=_log(rng, 9, 256), ny=2 * _log(rng, 8, 64),
                        p=rng.choice([2, 3, 4]))
        p = rng.choice([1, 2, 3, 3, 4])
        most = {1: 40, 2: 36, 3: 30, 4: 22}[p]
        return dict(kind="operator", flow=flow, nx=_log(rng, 3, most), ny=_log(rng, 3, most), nz=_log(rng, 3, most),
                    p=p, jv=rng.choice([0, 0, 0, 1]))
    if pick == "blocks":
        if flow == "vortex":
            p = rng.choice([2, 3, 3, 4])
            most = {2: 160, 3: 140, 4: 80}[p]
            return dict(kind="blocks", flow=flow, nx=_log(rng, 9, most), ny=_log(rng, 9, most), p=p,
                        precision=rng.choice([0, 0, 1, 2]), riemann=rng.choice([0, 1]))
        if flow == "channel":
            return dict(kind="blocks", flow=flow, nx=_log(rng, 9, 64), ny=2 * _log(rng, 8, 32), p=rng.choice([2, 3]),
                        precision=rng.choice([0, 1, 2]))
        p = rng.choice([1, 2, 3])
        most = {1: 16, 2: 10, 3: 12}[p]
        precision = rng.choice([0, 1, 2]) if p < 3 else rng.choice([1, 2])   # 320-row blocks: FP32 or BF16 only
        return dict(kind="blocks", flow=flow, nx=_log(rng, 3, most), ny=_log(rng, 3, most), nz=_log(rng, 3, most), p=p,
                    precision=precision, columns=1 if precision and rng.random() < 0.7 else 0)
    scheme = rng.choice(["row2", "row3", "row3", "row4", "bdf2", "esdirk2", "esdirk3", "ssprk3"])
    tol = 0.1 if scheme in ("bdf2", "esdirk2", "esdirk3") else rng.choice([1e-4, 1e-6, 1e-8])
    if flow == "vortex":
        most = 60 if scheme.startswith("esdirk") else 120
        nx, ny, p = _log(rng, 10, most), _log(rng, 10, most), rng.choice([2, 3, 3, 4])
        cfl = 0.1 if scheme == "ssprk3" else rng.uniform(4.0, 14.0)
        return dict(kind="step", flow=flow, scheme=scheme, nx=nx, ny=ny, p=p, precision=rng.choice([0, 0, 1, 2]),
                    riemann=rng.choice([0, 1]), jv=0, dt=round(cfl * 10.0 / max(nx, ny) / ((p + 1) * 4.2427), 6), tol=tol)
    scheme = rng.choice(["row2", "row3", "row4", "bdf2", "esdirk2"])
    tol = 0.1 if scheme in ("bdf2", "esdirk2") else 1e-6
    if flow == "channel":
        return dict(kind="step", flow=flow, scheme=scheme, nx=_log(rng, 10, 64), ny=2 * _log(rng, 8, 24),
                    p=rng.choice([2, 3]), precision=rng.choice([0, 1, 2]), riemann=0, jv=0, dt=1e-3, tol=tol)
    p = rng.choice([1, 2, 3])
    return dict(kind="step", flow=flow, scheme=scheme, nx=_log(rng, 4, 8), ny=_log(rng, 4, 8), nz=_log(rng, 4, 8), p=p,
                precision=rng.choice([1, 2]), columns=1, riemann=0, jv=rng.choice([0, 1]), dt=0.04, tol=tol)


# ------------------------------------------------------------------ inputs --

def _gen(seed, salt=0):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) * 1009 + salt)
    return g


def _edges(n, lo, hi, stretch, rng):
    e = np.linspace(lo, hi, n + 1)
    if stretch:
        e[1:-1] += rng.uniform(-stretch, stretch, n - 1) * (hi - lo) / n
    return e


def _wall_edges(ny):
    """Edges on [0, 1] clustered towards both walls: cells grow by 1.15 from 1e-3 (by more where
    that would not reach the centre) and are capped at the size that fills the rest."""
    half, first = ny // 2, 1e-3

    def sizes(ratio, cap):
        return np.minimum(first * ratio ** np.arange(half), cap)

    ratio, lo, hi = 1.15, first, 1.0
    if sizes(ratio, np.inf).sum() < 0.5:
        cap, lo, hi = np.inf, 1.15, 1e3
        for _ in range(200):
            ratio = 0.5 * (lo + hi)
            lo, hi = (ratio, hi) if sizes(ratio, np.inf).sum() < 0.5 else (lo, ratio)
    else:
        for _ in range(200):
            cap = 0.5 * (lo + hi)
            lo, hi = (cap, hi) if sizes(ratio, cap).sum() < 0.5 else (lo, cap)
    low = np.concatenate([[0.0], np.cumsum(sizes(ratio, cap))])
    low *= 0.5 / low[-1]
    return np.concatenate([low, 1.0 - low[-2::-1]])


def _mesh(case, seed):
    rng = np.random.default_rng(int(seed) + 77)
    if case["flow"] == "vortex":
        s = case.get("stretch", 0.0)
        return [_edges(case["nx"], -5.0, 5.0, s, rng), _edges(case["ny"], -5.0, 5.0, s, rng)]
    if case["flow"] == "channel":
        return [np.linspace(0.0, 2.0, case["nx"] + 1), _wall_edges(case["ny"])]
    return [np.linspace(-math.pi, math.pi, case[k] + 1) for k in ("nx", "ny", "nz")]


def _points(edges, p):
    """Coordinates of the Gauss-Legendre points of every element, each (Ne, Np)."""
    x, _ = np.polynomial.legendre.leggauss(p + 1)
    nd, n = len(edges), p + 1
    shape = [len(e) - 1 for e in reversed(edges)] + [n] * nd
    out = []
    for d, e in enumerate(edges):
        c = e[:-1, None] + 0.5 * (x[None, :] + 1.0) * np.diff(e)[:, None]
        view = [1] * (2 * nd)
        view[nd - 1 - d], view[2 * nd - 1 - d] = c.shape
        c = torch.from_numpy(c).cuda().reshape(view).expand(shape)
        out.append(c.reshape(-1, n ** nd))
    return out


def _conserved(rho, vel, pr):
    e = pr / (GAMMA - 1.0) + 0.5 * rho * sum(v * v for v in vel)
    return torch.stack([rho] + [rho * v for v in vel] + [e], dim=1).contiguous()


def _vortex(X, Y, alpha, theta, x0, y0, t=0.0):
    """Isentropic vortex of strength alpha in a free stream of speed sqrt(2), Mach 0.5."""
    ui, vi, pinf = math.sqrt(2.0) * math.cos(theta), math.sqrt(2.0) * math.sin(theta), 2.0 / (GAMMA * 0.25)
    dx, dy = X - x0 - ui * t, Y - y0 - vi * t
    dx, dy = dx - 10.0 * torch.round(dx / 10.0), dy - 10.0 * torch.round(dy / 10.0)
    ex = torch.exp(0.5 * (1.0 - dx * dx - dy * dy))
    T = pinf - alpha ** 2 * (GAMMA - 1.0) / (8.0 * GAMMA * math.pi ** 2) * ex * ex
    rho = (T / pinf) ** (1.0 / (GAMMA - 1.0))
    k = alpha / (2.0 * math.pi)
    return _conserved(rho, [ui - k * dy * ex, vi + k * dx * ex], rho * T)


def _state(case, edges, seed, t=0.0):
    rng = np.random.default_rng(int(seed))
    p = case["p"]
    if case["flow"] == "vortex":
        X, Y = _points(edges, p)
        x0, y0 = rng.uniform(-1.0, 1.0, 2)
        return _vortex(X, Y, rng.uniform(4.0, 5.0), math.pi / 4, x0, y0, t)
    if case["flow"] == "channel":
        # Poiseuille profile plus a divergence-free perturbation of 1e-2, at rest on the walls
        X, Y = _points(edges, p)
        w, dw = (Y * (1 - Y)) ** 2, 2 * Y * (1 - Y) * (1 - 2 * Y)
        up, vp = torch.zeros_like(X), torch.zeros_like(X)
        for _ in range(4):
            kx, a, ph = math.pi * rng.integers(1, 4), rng.uniform(0.2, 1.0), rng.uniform(0, 2 * math.pi)
            up += a * torch.sin(kx * X + ph) * dw
            vp -= a * kx * torch.cos(kx * X + ph) * w
        s = 1e-2 / up.abs().max()
        one = torch.ones_like(X)
        return _conserved(one, [4 * Y * (1 - Y) + s * up, s * vp], 25.0 / GAMMA * one)
    X, Y, Z = _points(edges, p)
    ph = rng.uniform(0, 2 * math.pi, 3)
    X, Y, Z = X + ph[0], Y + ph[1], Z + ph[2]
    p0 = 100.0 / GAMMA
    pr = p0 + (torch.cos(2 * X) + torch.cos(2 * Y)) * (torch.cos(2 * Z) + 2.0) / 16.0
    return _conserved(pr / p0, [torch.sin(X) * torch.cos(Y) * torch.cos(Z), -torch.cos(X) * torch.sin(Y) * torch.cos(Z),
                                torch.zeros_like(X)], pr)


def _gas(flow):
    if flow == "channel":
        return dict(mu=0.002, prandtl=0.72, body_force_x=0.016, wall_temperature=25.0 / GAMMA)
    if flow == "tgv":
        return dict(mu=1.0 / 1600.0, prandtl=0.71)
    return {}


def _context(case, edges, **kw):
    import paper_1904_04825_gb300 as fr
    opts = fr.default_opts(riemann=case.get("riemann", 0), jv_precision=case.get("jv", 0),
                           block_precision=case.get("precision", 0), block_columns=case.get("columns", 0),
                           **_gas(case["flow"]), **kw)
    if case["flow"] == "tgv":
        return fr.Context3D(*edges, case["p"], opts)
    return fr.Context(*edges, case["p"], opts, wall_y=case["flow"] == "channel")


def _instances(case, seed):
    """Meshes, degrees and vortex parameters of a batch: sizes and degrees from the case alone, flows from the seed."""
    rng, flow = np.random.default_rng(case["count"] * 131 + case["largest"]), np.random.default_rng(int(seed))
    lo, hi, out = math.log(case["smallest"]), math.log(case["largest"]), []
    for k in range(case["count"]):
        n, p = int(round(math.exp(lo + (hi - lo) * k / (case["count"] - 1)))), int(rng.integers(2, 5))
        x0, y0 = flow.uniform(-2.5, 2.5, 2)
        out.append((n, p, flow.uniform(3.0, 6.0), flow.uniform(0.0, 2 * math.pi), x0, y0))
    return out


def _net(case, seed):
    """He-uniform weights of the network 3 nb -> 256 -> 256 -> nb, flat [W1 b1 W2 b2 W3 b3]."""
    rng, sizes, flat = np.random.default_rng(int(seed)), [3 * case["nb"], 256, 256, case["nb"]], []
    for a, b in zip(sizes[:-1], sizes[1:]):
        lim = math.sqrt(6.0 / a)
        flat += [rng.uniform(-lim, lim, a * b).astype(np.float32), rng.uniform(-0.05, 0.05, b).astype(np.float32)]
    return sizes, flat


def _rows(case, seed):
    X = torch.randn(case["rows"], 3 * case["nb"], generator=_gen(seed, 1), device="cuda")
    T = torch.randn(case["rows"], case["nb"], generator=_gen(seed, 2), device="cuda")
    return X, T


# ---------------------------------------------------------- prepare and run --

def prepare(case, seed):
    import paper_1904_04825_gb300 as fr
    kind = case["kind"]
    if kind in ("train", "infer"):
        sizes, flat = _net(case, seed)
        X, T = _rows(case, seed)
        net = fr.MLP(sizes[0], sizes[1], sizes[3], case["rows"])
        net.set_params(np.concatenate(flat))
        return dict(case=case, net=net, X=X, T=T, Y=torch.empty_like(T))
    if kind == "batch":
        inst = _instances(case, seed)
        meshes = [(np.linspace(-5, 5, i[0] + 1), np.linspace(-5, 5, i[0] + 1)) for i in inst]
        batch = fr.Batch(meshes, [i[1] for i in inst],
                         fr.default_opts(tol_lin=case["tol"], block_precision=case["precision"]))
        U0 = [_vortex(*_points(m, i[1]), *i[2:]) for m, i in zip(meshes, inst)]
        return dict(case=case, batch=batch, U0=U0, U=[u.clone() for u in U0])
    edges = _mesh(case, seed)
    if kind == "step":
        ctx = _context(case, edges, tol_lin=case["tol"], precond=0 if case["scheme"] == "ssprk3" else 1)
        U0 = _state(case, edges, seed)
        P0 = _state(case, edges, seed, -case["dt"]) if case["scheme"] == "bdf2" else None
        return dict(case=case, ctx=ctx, U0=U0, U=U0.clone(), P0=P0, P=P0.clone() if P0 is not None else None,
                    ptc=fr.default_ptc_opts(tol_nl=1e-6, tol_lin=case["tol"]))
    U = _state(case, edges, seed)
    # a Krylov vector is rough on the scale of the points: normal entries
    z = torch.randn(U.shape, generator=_gen(seed), device="cuda", dtype=torch.float64)
    ctx = _context(case, edges, m_max=1, gmres_m=1, precond=1 if kind == "blocks" else 0)
    return dict(case=case, ctx=ctx, U=U, z=z, R=torch.empty_like(U), y=torch.empty_like(U))


def run(state):
    import paper_1904_04825_gb300 as fr
    case, kind = state["case"], state["case"]["kind"]
    if kind == "infer":
        state["net"].forward(state["X"], state["Y"], bf16=True)
        return {"Y": state["Y"]}
    if kind == "train":
        net = state["net"]
        net.forward(state["X"], state["Y"])
        loss = net.backward(state["X"], state["T"])
        net.adam(1e-3)
        return {"Y": state["Y"], "loss": loss, "params": net.get_params()}
    if kind == "batch":
        for u, u0 in zip(state["U"], state["U0"]):
            u.copy_(u0)
        state["batch"].step_row(4, case["dt"], state["U"])
        return {"U": state["U"]}
    ctx, U = state["ctx"], state["U"]
    if kind == "operator":
        fr.fr_residual(ctx, U, state["R"])
        fr.fr_jv(ctx, U, state["R"], state["z"], SHIFT, state["y"])
        return {"R": state["R"], "Az": state["y"]}
    if kind == "blocks":
        fr.ejacobi_factor(ctx, U, None, SHIFT)
        fr.ejacobi_apply(ctx, state["z"], state["y"])
        return {"z": state["y"]}
    scheme, dt = case["scheme"], case["dt"]
    U.copy_(state["U0"])
    if scheme == "ssprk3":
        fr.step_ssprk3(ctx, dt, U)
    elif scheme == "bdf2":
        state["P"].copy_(state["P0"])
        fr.step_bdf2(ctx, dt, U, state["P"], False, state["ptc"])
        return {"U": U, "U_prev": state["P"]}
    elif scheme.startswith("esdirk"):
        fr.step_esdirk(ctx, int(scheme[-1]), dt, U, state["ptc"])
    else:
        fr.step_row(ctx, int(scheme[-1]), dt, U)
    return {"U": U}


# -------------------------------------------------------------------- work --

def _residual_flops(flow, p):
    """Of one R(U) per element: fluxes at the points, traces, one common flux a face, corrected divergence."""
    n = p + 1
    if flow == "tgv":
        return 30 * n ** 4 + 240 * n ** 3 + 735 * n * n + n ** 3 * (260 + 30 * (n + 2))
    if flow == "channel":
        return 8 * n * n + 16 * n ** 3 + 96 * n * n + 32 * n + 344 * n + n * n * (144 + 16 * (n + 2))
    return 26 * n * n + 32 * n * n + 140 * n + 16 * n * n * (n + 2)


def work(case):
    kind = case["kind"]
    if kind in ("train", "infer"):
        rows, nb = case["rows"], case["nb"]
        params = 3 * nb * 256 + 256 * 256 + 256 * nb + 512 + nb
        gemm = 2.0 * rows * (3 * nb * 256 + 256 * 256 + 256 * nb)
        if kind == "infer":
            return dict(bytes=4.0 * rows * 4 * nb + 2.0 * params, flops=gemm)
        # forward, weight gradients, input gradients of two layers; weights and two moments in and out
        return dict(bytes=4.0 * rows * 5 * nb + 24.0 * params, flops=2 * gemm + 2.0 * rows * (256 * 256 + 256 * nb))
    if kind == "batch":
        parts = [dict(kind="step", flow="vortex", scheme="row4", nx=n, ny=n, p=p, precision=case["precision"],
                      tol=case["tol"]) for n, p, *_ in _instances(case, 0)]
        each = [work(c) for c in parts]
        return {k: sum(w[k] for w in each) for k in ("bytes", "flops")}
    flow, p = case["flow"], case["p"]
    ne = case["nx"] * case["ny"] * case.get("nz", 1)
    nb = 5 * (p + 1) ** 3 if flow == "tgv" else 4 * (p + 1) ** 2
    nd, per = ne * nb, _residual_flops(flow, p)
    if kind == "operator":
        return dict(bytes=(16.0 + 32.0) * nd, flops=(2.0 * per + 6.0 * nb) * ne)
    width = {0: 8, 1: 4, 2: 2}[case.get("precision", 0)]
    if kind == "blocks":
        # the blocks are written by the inversion and read by the apply
        return dict(bytes=(2.0 * width * nb + 24.0) * nd, flops=(2.0 * nb ** 3 + 2.0 * nb * nb) * ne)
    if case["scheme"] == "ssprk3":
        return dict(bytes=7 * 8.0 * nd, flops=3.0 * (per + 5 * nb) * ne)
    # stages of about 15 Arnoldi iterations each: blocks, A z and half of the basis twice
    solves = {"row2": 3, "row3": 4, "row4": 6, "bdf2": 2, "esdirk2": 8, "esdirk3": 12}[case["scheme"]]
    iters = 15.0 * solves
    return dict(bytes=iters * (width * nb + 24.0 + 32.0 + 160.0) * nd + 2.0 * width * nb * nd,
                flops=iters * (2.0 * nb * nb + per + 40.0 * nb) * ne + 2.0 * nb ** 3 * ne)


# ---------------------------------------------------- the same in 64 bits --
# The flux reconstruction in plain torch FP64.  Q: (var, [nz,] ny, nx, [k,] j, i); direction d has the
# element axis nd - d and the point axis 2 nd - d; a face array lacks that point axis.

class _Fr:
    def __init__(self, case, edges):
        self.nd, self.p, self.flow = len(edges), case["p"], case["flow"]
        self.n, self.roe = self.p + 1, case.get("riemann", 0) == 1
        self.wall = self.flow == "channel"
        gas = _gas(self.flow)
        self.mu, self.force, self.tw = gas.get("mu", 0.0), gas.get("body_force_x", 0.0), gas.get("wall_temperature", 1.0)
        self.kappa = self.mu * GAMMA / (GAMMA - 1.0) / gas["prandtl"] if self.mu else 0.0
        self.nel = [len(e) - 1 for e in reversed(edges)]
        self.h = []
        for d, e in enumerate(edges):
            view = [1] * (2 * self.nd + 1)
            view[self.nd - d] = len(e) - 1
            self.h.append(torch.from_numpy(np.diff(e)).cuda().reshape(view))
        x, _ = np.polynomial.legendre.leggauss(self.n)
        L = np.polynomial.legendre
        basis = [np.poly1d(np.poly([v for j, v in enumerate(x) if j != k])) for k in range(self.n)]
        basis = [b / b(x[k]) for k, b in enumerate(basis)]
        c = np.zeros(self.n + 1)
        c[self.n], c[self.n - 1] = 1.0, -1.0
        dgl = L.legval(x, L.legder(c * (-1.0) ** self.n / 2))
        dgr = -L.legval(-x, L.legder(c * (-1.0) ** self.n / 2))
        t = lambda a: torch.tensor(np.array(a), dtype=torch.float64, device="cuda")  # noqa: E731
        self.D = t([[b.deriv()(v) for b in basis] for v in x])
        self.ends = [t([b(s) for b in basis]) for s in (-1.0, 1.0)]
        self.dg = [t(dgl), t(dgr)]

    def grid(self, U):
        nv = U.shape[1]
        return U.reshape(*self.nel, nv, *([self.n] * self.nd)).movedim(self.nd, 0)

    def flat(self, Q):
        return Q.movedim(0, self.nd).reshape(-1, Q.shape[0], self.n ** self.nd).contiguous()

    def along(self, M, x, d):
        return (x.movedim(2 * self.nd - d, -1) @ M.T).movedim(-1, 2 * self.nd - d)

    def trace(self, x, d, side):
        return x.movedim(2 * self.nd - d, -1) @ self.ends[side]

    def lift(self, f, d, side):
        view = [1] * (2 * self.nd + 1)
        view[2 * self.nd - d] = self.n
        return f.unsqueeze(2 * self.nd - d) * self.dg[side].reshape(view)

    def flux(self, q, d):
        un = q[1 + d] / q[0]
        pr = (GAMMA - 1.0) * (q[-1] - 0.5 * sum(q[1 + c] ** 2 for c in range(self.nd)) / q[0])
        f = [q[1 + d]] + [q[1 + c] * un + (pr if c == d else 0.0) for c in range(self.nd)] + [un * (q[-1] + pr)]
        return torch.stack(f), un, pr

    def viscous(self, q, g, d):
        nd, v = self.nd, [q[1 + c] / q[0] for c in range(self.nd)]
        dv = [[(g[c][1 + m] - v[m] * g[c][0]) / q[0] for m in range(nd)] for c in range(nd)]
        dT = (GAMMA - 1.0) * ((g[d][-1] - q[-1] / q[0] * g[d][0]) / q[0] - sum(v[m] * dv[d][m] for m in range(nd)))
        div = sum(dv[c][c] for c in range(nd))
        tau = [self.mu * (dv[d][m] + dv[m][d] - (2.0 / 3.0 * div if m == d else 0.0)) for m in range(nd)]
        return torch.stack([torch.zeros_like(div)] + tau + [sum(v[m] * tau[m] for m in range(nd)) + self.kappa * dT])

    def common(self, qm, qp, d):
        (fm, um, pm), (fp, up, pp) = self.flux(qm, d), self.flux(qp, d)
        if not self.roe:
            lam = torch.maximum(um.abs() + (GAMMA * pm / qm[0]).sqrt(), up.abs() + (GAMMA * pp / qp[0]).sqrt())
            return 0.5 * (fm + fp) - 0.5 * lam * (qp - qm)
        sm, sp = qm[0].sqrt(), qp[0].sqrt()
        mean = lambda a, b: (sm * a + sp * b) / (sm + sp)  # noqa: E731
        v = [mean(qm[1 + c] / qm[0], qp[1 + c] / qp[0]) for c in range(2)]
        H = mean((qm[-1] + pm) / qm[0], (qp[-1] + pp) / qp[0])
        k, rho, un, t = 0.5 * (v[0] ** 2 + v[1] ** 2), sm * sp, v[d], 1 - d
        a2 = (GAMMA - 1.0) * (H - k)
        a, dp, du = a2.sqrt(), pp - pm, up - um
        l1, l4 = (un - a).abs() * (dp - rho * a * du) / (2 * a2), (un + a).abs() * (dp + rho * a * du) / (2 * a2)
        l2 = un.abs() * (qp[0] - qm[0] - dp / a2)
        l3 = un.abs() * rho * (qp[1 + t] / qp[0] - qm[1 + t] / qm[0])
        diss = [l1 + l2 + l4, None, None, l1 * (H - un * a) + l2 * k + l3 * v[t] + l4 * (H + un * a)]
        diss[1 + d], diss[1 + t] = l1 * (un - a) + l2 * un + l4 * (un + a), (l1 + l2 + l4) * v[t] + l3
        return 0.5 * (fm + fp) - 0.5 * torch.stack(diss)

    def traces(self, Q):
        """Per direction and side: the trace of the state and those of its gradient."""
        g = [2.0 / self.h[c] * self.along(self.D, Q, c) for c in range(self.nd)] if self.mu else []
        return [[[self.trace(x, d, s) for x in [Q] + g] for s in (0, 1)] for d in range(self.nd)]

    def seen(self, tr):
        """What each element's neighbours present to it on its low and high faces."""
        return [[[torch.roll(x, 1 - 2 * s, self.nd - d) for x in tr[d][1 - s]] for s in (0, 1)] for d in range(self.nd)]

    def residual(self, Q, nbr=None):
        nd, own, br2 = self.nd, self.traces(Q), (self.p + 1) * (self.p + 2) / 2.0
        nbr = nbr if nbr is not None else self.seen(own)
        qc, fn = [[None, None] for _ in range(nd)], [[None, None] for _ in range(nd)]
        for d in range(nd):
            h = self.h[d].squeeze(2 * nd - d)
            for s in (0, 1):
                o, x = own[d][s], nbr[d][s]
                m, pl = (x, o) if s == 0 else (o, x)
                ho = torch.roll(h, 1 - 2 * s, nd - d)
                hm, hp = (ho, h) if s == 0 else (h, ho)
                c, f = 0.5 * (m[0] + pl[0]), self.common(m[0], pl[0], d)
                if self.mu:
                    g = [0.5 * (m[1 + k] + pl[1 + k]) for k in range(nd)]
                    g[d] = g[d] + 0.5 * (2.0 / hm * br2 * (c - m[0]) - 2.0 / hp * br2 * (c - pl[0]))
                    f = f - self.viscous(c, g, d)
                if self.wall and d == 1:
                    at = (slice(None), 0 if s == 0 else -1)
                    q = o[0][at]
                    w = torch.stack([q[0], 0 * q[0], 0 * q[0], q[0] * self.tw / (GAMMA - 1.0)])
                    sign = -1.0 if s == 0 else 1.0
                    gw = [o[1][at], o[2][at] + sign * 2.0 / h[at] * br2 * (w - q)]
                    c[at], f[at] = w, self.flux(w, 1)[0] - self.viscous(w, gw, 1)
                qc[d][s], fn[d][s] = c, f
        if self.mu:
            g = [2.0 / self.h[c] * (self.along(self.D, Q, c) + sum(self.lift(qc[c][s] - own[c][s][0], c, s) for s in (0, 1)))
                 for c in range(nd)]
        R = torch.zeros_like(Q)
        for d in range(nd):
            F = self.flux(Q, d)[0] - (self.viscous(Q, g, d) if self.mu else 0.0)
            R -= 2.0 / self.h[d] * (self.along(self.D, F, d) + sum(self.lift(fn[d][s] - self.trace(F, d, s), d, s) for s in (0, 1)))
        if self.force:
            R[1] += self.force * Q[0]
            R[3] += self.force * Q[1]
        return R


def _exact_net(case, seed):
    sizes, flat = _net(case, seed)
    X, T = (t.double() for t in _rows(case, seed))
    P = [torch.from_numpy(a).cuda().double() for a in flat]
    W = [P[2 * k].reshape(sizes[k + 1], sizes[k]) for k in range(3)]
    A, Z = [X], []
    for k in range(3):
        Z.append(A[-1] @ W[k].T + P[2 * k + 1])
        A.append(Z[-1].clamp(min=0.0))
    if case["kind"] == "infer":
        return {"Y": Z[2]}
    d, new = (Z[2] - T) / Z[2].numel(), [None] * 6
    for k in (2, 1, 0):
        for i, g in ((2 * k, d.T @ A[k]), (2 * k + 1, d.sum(0))):
            # the first Adam step: both moments corrected for their bias are g and g^2
            new[i] = P[i] - 1e-3 * g.reshape(-1) / (g.reshape(-1).abs() + 1e-8)
        if k:
            d = (d @ W[k]) * (Z[k - 1] > 0)
    return {"Y": Z[2], "loss": float(0.5 * (Z[2] - T).square().mean()), "params": torch.cat(new)}


def exact(case, seed):
    kind = case["kind"]
    if kind in ("train", "infer"):
        return _exact_net(case, seed)
    if kind == "batch" or (kind == "step" and case["scheme"] != "ssprk3"):
        return None   # a whole implicit step: iterative solves stopped at a tolerance
    edges = _mesh(case, seed)
    U, op = _state(case, edges, seed), _Fr(case, edges)
    Q = op.grid(U)
    if kind == "step":
        dt = case["dt"]
        q1 = Q + dt * op.residual(Q)
        q2 = 0.75 * Q + 0.25 * (q1 + dt * op.residual(q1))
        return {"U": op.flat(Q / 3.0 + 2.0 / 3.0 * (q2 + dt * op.residual(q2)))}
    z = torch.randn(U.shape, generator=_gen(seed), device="cuda", dtype=torch.float64)
    if kind == "operator":
        R = op.residual(Q)
        eps = 1e-7 * (1.0 + U.norm()) / z.norm()
        Az = SHIFT * z - op.flat(op.residual(Q + eps * op.grid(z)) - R) / eps
        return {"R": op.flat(R), "Az": Az}
    # blocks: element-local forward differences with the neighbours' traces kept
    nb, nbr = U.shape[1] * U.shape[2], op.seen(op.traces(Q))
    R, M = op.residual(Q, nbr), torch.empty(U.shape[0], nb, nb, dtype=torch.float64, device="cuda")
    for c in range(nb):
        V = U.clone()
        col = V.view(-1, nb)[:, c]
        step = 1e-7 * (1.0 + col.abs())
        col += step
        M[:, :, c] = -op.flat(op.residual(op.grid(V), nbr) - R).view(-1, nb) / step[:, None]
    M.diagonal(dim1=1, dim2=2).add_(SHIFT)
    return {"z": torch.linalg.solve(M, z.view(-1, nb)).view(U.shape)}
