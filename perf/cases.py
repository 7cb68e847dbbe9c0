"""Workloads of the framework's public entry points, for timing and for comparing outputs.

Four kinds of case:

* ``step``  -- one lattice: initial density on the device -> ``Context.set_density_device``,
  ``Context.step(steps)``, and the populations (``Context.device_populations``).  Both models, both
  precisions, periodic lattices and walled channels, the droplet-collision drive and the full
  free-energy model (A != 0);
* ``sweep`` -- a batch of uneven calibration lattices: ``Batch.run`` and ``Batch.observables``;
* ``train`` -- full-batch training of the calibration surrogate: ``Surrogate.set_params``,
  ``Surrogate.train``, ``Surrogate.params``;
* ``query`` -- inference of the surrogate on device arrays: ``Surrogate.predict_device``.

Runs of the framework take 5e3 to 1e5 steps (or 6e4 training iterations); a pass here takes a few
hundred, which is the same work per step in a shorter pass.
"""
import math

import numpy as np
import torch

from paper_2403_11167_gb300 import lbm

PP, FE = 0, 1

# Carnahan-Starling constants and the pseudopotential's consistency parameter of the droplet tests
# (eps = 1.9168): given by the case, so that a reference needs no quadrature of the model's theory.
A_EOS, B_EOS, SIGMA_LI = 0.25, 4.0, 1.9168 / 16.0


def _step(name, model, prec, nx, ny, steps, scene, Tr=0.8, tau=1.0, walls=0, drive=0.0, A=0.0):
    c = dict(kind="step", model=model, precision=prec, nx=nx, ny=ny, steps=steps, scene=scene, Tr=Tr, tau=tau,
             walls=walls, drive=drive, A=A)
    return dict(c, name=name) if name else c


def listed():
    return [
        # the throughput configuration: spinodal decomposition on 4096 x 4096, both models, FP32
        _step("pp_f32_4096", PP, 32, 4096, 4096, 64, "spinodal", Tr=0.85, tau=0.8),
        _step("fe_f32_4096", FE, 32, 4096, 4096, 64, "spinodal", Tr=0.85, tau=0.8),
        # the static-droplet (Laplace) configuration: 256 x 256, FP32, thousands of short steps
        _step("fe_f32_droplet_256", FE, 32, 256, 256, 512, "droplet"),
        # a mid-size lattice whose width is not a multiple of 4
        _step("pp_f32_ragged_1022x770", PP, 32, 1022, 770, 128, "spinodal", Tr=0.85, tau=0.8),
        # the flat-interface configuration: 256 x 4, FP64 (the smallest lattice)
        _step("pp_f64_slab_256x4", PP, 64, 256, 4, 512, "slab"),
        # the flow between parallel plates of Sec. 5.3: 101 x 50, no-slip walls, body force, FP64
        _step("fe_f64_channel_101x50", FE, 64, 101, 50, 256, "channel", walls=1),
        # the droplet collision of Sec. 5.4: 200 x 100, density-dependent drive, FP64
        _step("pp_f64_collision_200x100", PP, 64, 200, 100, 256, "pair", drive=5e-6),
        # the full free-energy model (viscosity-tuning term), FP32
        _step("fe_f32_full_A_1024", FE, 32, 1024, 1024, 128, "droplet", A=0.15),
        # the calibration sweep: slabs 64 x 4 .. 512 x 4 and droplets 64^2 .. 512^2 in one batch
        dict(name="sweep_96", kind="sweep", lattices=96, shapes=11167, min_steps=100, max_steps=400),
        # training the surrogate on the size of its real training set
        dict(name="train_8000", kind="train", sets=7973, iterations=24),
        # surrogate queries: one calibration request batch, and a dense parameter scan
        dict(name="query_4096", kind="query", queries=4096, mode=0),
        dict(name="query_262144", kind="query", queries=262144, mode=0),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the same ranges."""
    kind = rng.choice(["f32", "f32", "f32", "f32", "f64", "f64", "sweep", "train", "query"])
    model = rng.choice([PP, FE])
    Tr, tau = round(rng.uniform(0.75, 0.9), 3), round(rng.uniform(0.7, 1.1), 3)
    if kind in ("f32", "f64"):
        prec = int(kind[1:])
        # FP32: 64 x 8 .. 4096 x 4096; FP64 (parity and flow tests): 64 x 4 .. 400 x 300
        nx = _log(rng, 64, 4096) if prec == 32 else _log(rng, 64, 400)
        ny = _log(rng, 8, 4096) if prec == 32 else _log(rng, 4, 300)
        if prec == 32 and rng.random() < 0.7:
            nx -= nx % 4  # most FP32 lattices are a multiple of 4 wide
        option = rng.choice(["", "", "walls", "drive", "A"])
        walls = 1 if option == "walls" and ny >= 6 else 0
        drive = 5e-6 if option == "drive" else 0.0
        A = round(rng.uniform(-0.1, 0.15), 3) if option == "A" and model == FE else 0.0
        scene = "channel" if walls else "pair" if drive else rng.choice(["spinodal", "droplet", "slab"])
        # as many steps as keep the pass at or under that of the largest listed lattice
        steps = max(16, min(rng.randint(192, 640), int(2.5e8 if prec == 32 else 5e6) // (nx * ny)))
        return _step(None, model, prec, nx, ny, steps, scene, Tr, tau, walls, drive, A)
    if kind == "sweep":
        return dict(kind="sweep", lattices=rng.randint(8, 128), shapes=rng.randint(1, 1 << 20),
                    min_steps=rng.randint(50, 100), max_steps=rng.randint(150, 300))
    if kind == "train":
        return dict(kind="train", sets=_log(rng, 200, 7973), iterations=rng.randint(8, 24))
    return dict(kind="query", queries=_log(rng, 1, 262144), mode=rng.choice([0, 0, 1]))


# ---------------------------------------------------------------------------------------
# Thermodynamics of the Carnahan-Starling EOS (Eq. 28) in plain numpy.  With e = b rho / 4 and
# alpha = 4 a / (b R T):  p b / (4 R T) = Z(e) - alpha e^2, Z(e) = e (1 + e + e^2 - e^3) / (1 - e)^3,
# and mu_b / (R T) = (3 - e) / (1 - e)^3 + ln e - 2 alpha e + const.

_N = np.polynomial.Polynomial([1.0, 4.0, 4.0, -4.0, 1.0])  # Z'(e) = N(e) / (1 - e)^4
_U = np.polynomial.Polynomial([1.0, -1.0])                 # 1 - e
_E = np.polynomial.Polynomial([0.0, 1.0])


def _critical_RT(a, b):
    """R T_c: Z' R T = 8 a e / b and Z'' R T = 8 a / b, i.e. e Z'' = Z'."""
    g = _E * (_N.deriv() * _U + 4.0 * _N) - _N * _U
    lo, hi = 0.05, 0.3
    for _ in range(100):
        m = 0.5 * (lo + hi)
        lo, hi = (lo, m) if (g(m) > 0) == (g(hi) > 0) else (m, hi)
    e = 0.5 * (lo + hi)
    return 8.0 * a * e * (1.0 - e) ** 4 / (b * _N(e))


def _real_roots(poly):
    r = poly.roots()
    return sorted(float(x.real) for x in r if abs(x.imag) < 1e-9 and 0.0 < x.real < 0.999)


def _coexistence(a, b, Tr):
    """(rho_v, rho_l) with equal pressure and chemical potential (bulk values of the initial fields)."""
    alpha = 4.0 * a / (b * Tr * _critical_RT(a, b))
    spin = _real_roots(_N - 2.0 * alpha * _E * _U ** 4)
    Z = lambda e: e * (1 + e + e * e - e ** 3) / (1 - e) ** 3 - alpha * e * e  # noqa: E731
    mu = lambda e: (3 - e) / (1 - e) ** 3 + math.log(e) - 2 * alpha * e        # noqa: E731
    ends = lambda q: _real_roots(_E * (1 + _E + _E ** 2 - _E ** 3) - (alpha * _E ** 2 + q) * _U ** 3)  # noqa: E731
    lo, hi = max(Z(spin[1]), 0.0) + 1e-12, Z(spin[0]) - 1e-12
    for _ in range(60):
        q = 0.5 * (lo + hi)
        r = ends(q)
        lo, hi = (lo, q) if mu(r[-1]) < mu(r[0]) else (q, hi)  # the denser phase favoured: pressure too high
    return 4.0 * r[0] / b, 4.0 * r[-1] / b


# ---------------------------------------------------------------------------------------
# Inputs


_STREAM = None


def _stream():
    """The program's stream: one for all contexts, as a user's program has."""
    global _STREAM
    if _STREAM is None:
        _STREAM = torch.cuda.Stream()
    return _STREAM


def _device():
    return "cuda" if torch.cuda.is_available() else "cpu"


def _density(case, seed):
    """Initial density (float64 tensor [ny, nx]) of a ``step`` case: the paper's scenes with the seed
    moving the centre, the radius or the noise."""
    nx, ny, dev = case["nx"], case["ny"], _device()
    rv, rl = _coexistence(A_EOS, B_EOS, case["Tr"])
    g = torch.Generator(device=dev).manual_seed(seed)
    r = np.random.default_rng(seed).uniform(-1.0, 1.0, 4)
    y, x = (torch.arange(n, dtype=torch.float64, device=dev) for n in (ny, nx))
    y = y[:, None]
    scene = case["scene"]
    if scene == "spinodal":
        noise = torch.rand((ny, nx), dtype=torch.float64, device=dev, generator=g) * 0.02 - 0.01
        return 0.5 * (rl + rv) * (1.0 + noise)
    if scene == "slab":
        s = 0.02 * nx * r[0]
        return (rv + 0.5 * (rl - rv) * (torch.tanh(0.4 * (x - nx / 4 - s)) - torch.tanh(0.4 * (x - 3 * nx / 4 - s)))
                ).expand(ny, nx).contiguous()
    if scene == "channel":  # vapour below, liquid above, a gently wavy interface
        h = 0.5 * (ny - 1) + 0.05 * ny * r[0] + 0.02 * ny * torch.sin(2 * math.pi * x / nx + r[1])
        return rv + 0.5 * (rl - rv) * (1.0 + torch.tanh(0.4 * (y - h)))
    centres = [(0.5, 0.5)] if scene == "droplet" else [(0.25, 0.5), (0.75, 0.5)]
    rho = torch.full((ny, nx), rv, dtype=torch.float64, device=dev)
    R = (0.23 if scene == "droplet" else 0.18) * min(nx, ny) * (1.0 + 0.1 * r[3])
    for fx, fy in centres:
        d = torch.sqrt((x - fx * (nx - 1) - r[0]) ** 2 + (y - fy * (ny - 1) - r[1]) ** 2)
        rho = rho + 0.5 * (rl - rv) * (1.0 - torch.tanh(0.4 * (d - R)))
    return rho


def _body(case):
    return 1e-6 if case["walls"] else 0.0  # the channel's flow is driven by a constant body force


def _sweep(case, seed):
    """The lattices of a ``sweep`` case: half slabs nx x 4, half droplets L x L (uneven sizes and step
    counts from ``shapes``), temperatures, widths and relaxation times from the seed."""
    s, r = np.random.default_rng(case["shapes"]), np.random.default_rng(seed)
    out = []
    for i in range(case["lattices"]):
        flat = i % 2 == 0
        nx = int(s.choice([64, 128, 256, 512] if flat else [64, 128, 192, 256, 384, 512]))
        ny = 4 if flat else nx
        steps = int(s.integers(case["min_steps"], case["max_steps"] + 1))
        R = float(r.uniform(0.15, 0.28) * nx)
        Tr, kP, tau = float(r.uniform(0.65, 0.9)), float(r.choice([0.7, 1.0])), float(r.uniform(0.7, 1.1))
        rv, rl = _coexistence(A_EOS, B_EOS, Tr)
        x = np.arange(nx, dtype=np.float64)
        if flat:
            rho = rv + 0.5 * (rl - rv) * (np.tanh(0.4 * (x - nx / 4)) - np.tanh(0.4 * (x - 3 * nx / 4)))
            rho = np.ascontiguousarray(np.broadcast_to(rho, (ny, nx)))
        else:
            d = np.hypot(x - 0.5 * (nx - 1), x[:, None] - 0.5 * (ny - 1))
            rho = 0.5 * (rl + rv) - 0.5 * (rl - rv) * np.tanh(0.4 * (d - R))
        out.append(dict(nx=nx, ny=ny, geometry=0 if flat else 1, nsteps=steps, Tr=Tr, kappa_P=kP, tau=tau, rho=rho))
    return out


DIMS = (4, 128, 128, 128, 4)


def _network(seed):
    """A network as training leaves it in scale: weights of variance 2 / fan-in (the last layer small),
    small biases; and the standardisation of the calibration ranges."""
    r = np.random.default_rng(seed)
    parts = []
    for l in range(4):
        parts.append(r.normal(0.0, math.sqrt((2.0 if l < 3 else 0.5) / DIMS[l]), DIMS[l + 1] * DIMS[l]))
        parts.append(r.uniform(-0.1, 0.1, DIMS[l + 1]))
    stats = np.array([0.725, 0.375, 4.0, 0.7, 0.13, 0.072, 0.577, 0.245,
                      0.25, -5.0, 9.0, 0.008, 0.06, 1.0, 4.0, 0.004], dtype=np.float32)
    return np.concatenate(parts).astype(np.float32), stats


def _parameter_sets(n, seed):
    """Network inputs (Tr, a, b, kappa_P) over the calibration ranges and a smooth map like the
    calibrated observables; a third of the surface tensions missing, as kappa_P = 0.4 sets lack them."""
    r = np.random.default_rng(seed)
    X = np.column_stack([r.uniform(0.5, 0.95, n), r.uniform(0.25, 0.5, n), r.uniform(3, 5, n),
                         r.choice([0.4, 0.7, 1.0], n)])
    Y = np.column_stack([(1.3 - X[:, 0]) / X[:, 2], np.exp(-12 * (1 - X[:, 0]) ** 0.8) / X[:, 2],
                         3 + 6 * np.sqrt(X[:, 3]) / (1.05 - X[:, 0]), 0.04 * X[:, 1] * (1 - X[:, 0]) ** 1.5])
    Y[X[:, 3] == 0.4, 3] = np.nan
    return X.astype(np.float32), Y.astype(np.float32)


LR = 2e-3


def prepare(case, seed):
    kind = case["kind"]
    if kind == "step":
        prec = lbm.LBM_F64 if case["precision"] == 64 else lbm.LBM_F32
        p = lbm.lbm_params_default(case["model"], precision=prec, a=A_EOS, b=B_EOS, Tr=case["Tr"], tau_nu=case["tau"],
                                   A=case["A"], body_fx=_body(case))
        if case["model"] == PP:
            p.sigma_Li = SIGMA_LI
        ctx = lbm.Context(p, case["nx"], case["ny"], stream=_stream(), walls=bool(case["walls"]))
        if case["drive"]:
            ctx.set_drive(case["drive"], -case["drive"], case["nx"] // 2, -1)
        rho = _density(case, seed).to(torch.float64 if prec == lbm.LBM_F64 else torch.float32)
        torch.cuda.synchronize()
        return dict(case, ctx=ctx, rho=rho)
    if kind == "sweep":
        specs, rhos = [], []
        for e in _sweep(case, seed):
            p = lbm.lbm_params_default(PP, precision=lbm.LBM_F32, a=A_EOS, b=B_EOS, Tr=e["Tr"], tau_nu=e["tau"],
                                       kappa_P=e["kappa_P"], sigma_Li=SIGMA_LI)
            specs.append(dict(nx=e["nx"], ny=e["ny"], geometry=e["geometry"], nsteps=e["nsteps"], params=p))
            rhos.append(e["rho"])
        return dict(case, batch=lbm.Batch(specs, rhos))
    theta, stats = _network(seed)
    n = case["sets"] if kind == "train" else case["queries"]
    X, Y = _parameter_sets(n, seed + 1)
    if kind == "train":
        m = lbm.Surrogate(lbm.Surrogate.standardisation(X, Y), seed=0)
        return dict(case, m=m, theta=theta, X=X, Y=Y)
    m = lbm.Surrogate(stats, seed=0)
    m.set_params(theta)
    Xd = torch.from_numpy(X).cuda()
    return dict(case, m=m, X=Xd, Y=torch.empty_like(Xd))


def _populations(ctx, precision):
    """The current populations [9, ny, nx] as a view of the context's device memory."""
    ptr, pitch = ctx.device_populations()
    size = 8 if precision == 64 else 4
    off = ptr - ctx.workspace.data_ptr()
    f = ctx.workspace[off:off + 9 * pitch * size].view(torch.float64 if precision == 64 else torch.float32)
    return f.view(9, pitch)[:, :ctx.nx * ctx.ny].view(9, ctx.ny, ctx.nx)


OBSERVABLES = ("rho_l", "rho_v", "width", "dp", "u_max", "mass", "radius")


def run(state):
    kind = state["kind"]
    if kind == "step":
        ctx = state["ctx"]
        ctx.set_density_device(state["rho"])
        ctx.step(state["steps"])
        return _populations(ctx, state["precision"])
    if kind == "sweep":
        b = state["batch"]
        b.run()
        obs = b.observables()
        # numbers of an FP32 run, so given in that type
        return {k: np.array([o[k] for o in obs], dtype=np.float32) for k in OBSERVABLES}
    if kind == "train":
        m = state["m"]
        m.set_params(state["theta"])
        loss = m.train(state["X"], state["Y"], iterations=state["iterations"], lr=LR, lr_min=LR / 100)
        return {"loss": np.float32(loss), "params": m.params()}
    state["m"].predict_device(state["X"], state["Y"], stream=_stream().cuda_stream, mode=state["mode"])
    return state["Y"]


def work(case):
    kind = case["kind"]
    if kind == "step":
        # every step reads and writes nine populations per cell (FP32: and the int16 rest extension)
        n = case["nx"] * case["ny"] * case["steps"]
        return {"bytes": n * (144 if case["precision"] == 64 else 76), "flops": n * (250 if case["model"] == PP else 240)}
    if kind == "sweep":
        n = sum(e["nx"] * e["ny"] * e["nsteps"] for e in _sweep(case, 0))
        return {"bytes": n * 76, "flops": n * 250}
    w = sum(a * b for a, b in zip(DIMS, DIMS[1:]))
    if kind == "train":
        n, it = case["sets"], case["iterations"]
        # per iteration: forward, and the two products of the backward pass; the parameters, their
        # gradient and both moments; the samples
        return {"bytes": it * (4 * 34180 * 7 + n * 32), "flops": it * n * 6 * w}
    n = case["queries"]
    return {"bytes": n * 32 + 4 * 34180, "flops": n * 2 * w * (3 if case["mode"] == 0 else 1)}


# ---------------------------------------------------------------------------------------
# The same results in 64 bits, plain torch

CX = (0, 1, 0, -1, 0, 1, -1, -1, 1)
CY = (0, 0, 1, 0, -1, 1, 1, -1, -1)
W = (4 / 9,) + (1 / 9,) * 4 + (1 / 36,) * 4


def _moment_rows():
    c2 = [x * x + y * y for x, y in zip(CX, CY)]
    return [[1.0] * 9, [-4.0 + 3 * c for c in c2], [4.0 - 10.5 * c + 4.5 * c * c for c in c2],
            list(map(float, CX)), [x * (-5.0 + 3 * c) for x, c in zip(CX, c2)],
            list(map(float, CY)), [y * (-5.0 + 3 * c) for y, c in zip(CY, c2)],
            [float(x * x - y * y) for x, y in zip(CX, CY)], [float(x * y) for x, y in zip(CX, CY)]]


def _at(a, dx, dy, walls):
    """a at x + (dx, dy): periodic in x; in y periodic, or mirrored through wall nodes."""
    if dx:
        a = torch.roll(a, -dx, -1)
    if dy and walls:
        a = torch.cat([a[..., 1:, :], a[..., -2:-1, :]], -2) if dy > 0 else torch.cat([a[..., 1:2, :], a[..., :-1, :]], -2)
    elif dy:
        a = torch.roll(a, -dy, -2)
    return a


def _grad(a, walls):
    """Gradient of Eq. (24), 3 sum_i w_i a(x + c_i) c_i (equally the force stencil of Eq. 10)."""
    gx = gy = 0
    for i in range(1, 9):
        n = _at(a, CX[i], CY[i], walls)
        gx, gy = gx + 3 * W[i] * CX[i] * n, gy + 3 * W[i] * CY[i] * n
    return gx, gy


class _Reference:
    """Eq. (1) with the model's force, equilibrium, forcing and source, in moments (Eqs. S48, S49)."""

    def __init__(self, model, RT, tau, kappa_P=1.0, walls=0, drive=0.0, split=0, A=0.0, fx=0.0):
        self.model, self.RT, self.walls, self.drive, self.split, self.A, self.fx = model, RT, walls, drive, split, A, fx
        self.te, self.tz, self.tq, self.tn = ((tau, tau, 1 / 1.99, tau) if model == PP else
                                              (0.25 + 0.5 * tau, 1.0, 1.0, tau))
        self.kP, self.li = kappa_P, 12.0 * kappa_P * SIGMA_LI
        dev = _device()
        self.M = torch.tensor(_moment_rows(), dtype=torch.float64, device=dev)
        self.Mi = torch.linalg.inv(self.M.cpu()).to(dev)

    def init(self, rho):
        if self.model == PP:
            return torch.stack([w * rho for w in W])
        return torch.stack([rho] + [torch.zeros_like(rho)] * 8)

    def _pressure(self, rho):
        e = 0.25 * B_EOS * rho
        return rho * self.RT * (1 + e + e * e - e ** 3) / (1 - e) ** 3 - A_EOS * rho * rho

    def _mu(self, rho):
        e = 0.25 * B_EOS * rho
        bulk = self.RT * ((3 - e) / (1 - e) ** 3 + torch.log(rho)) - 2 * A_EOS * rho
        lap = 0
        for i in range(1, 9):
            lap = lap + 6 * W[i] * (_at(rho, CX[i], CY[i], self.walls) - rho)
        return bulk - 0.5 * lap

    def _fill(self, f, Jx):
        """Zou-He completion of the wall rows for the node momentum (Jx, 0)."""
        f1, f3 = f[1], f[3]
        h0, h1 = 0.5 * (f1[0] - f3[0]), 0.5 * (f1[-1] - f3[-1])
        f[2][0], f[5][0], f[6][0] = f[4][0], f[7][0] - h0 + 0.5 * Jx[0], f[8][0] + h0 - 0.5 * Jx[0]
        f[4][-1], f[7][-1], f[8][-1] = f[2][-1], f[5][-1] + h1 - 0.5 * Jx[-1], f[6][-1] - h1 + 0.5 * Jx[-1]

    def collide(self, f):
        """Populations after the collision, at the cells they leave."""
        walls = self.walls
        if walls:
            self._fill(f, torch.zeros_like(f[0]))
        rho = f.sum(0)
        fx = self.fx
        if self.drive:
            x = torch.arange(rho.shape[-1], dtype=torch.float64, device=rho.device)
            ax = self.drive * (1.0 - 2.0 * (x > self.split))
            fx = fx + ax * (rho - rho.mean()).abs()
        Qxx = Qyy = Qxy = L = 0
        if self.model == PP:
            psi = torch.sqrt(2 * (rho / 3 - self._pressure(rho)))
            Sx, Sy = _grad(psi, walls)
            Fx, Fy = psi * Sx + fx, psi * Sy
            L = self.li * (Sx * Sx + Sy * Sy)
            # Eq. (30), G = -1: C = G [C1 delta + C2 (c c - delta / 3)]
            C1, C2 = 5 / 6 * (self.kP - 1), 0.5 * (1 - self.kP)
            for i in range(1, 9):
                d = psi * 3 * W[i] * (_at(psi, CX[i], CY[i], walls) - psi)
                Qxx = Qxx - (C1 - C2 / 3 + C2 * CX[i] * CX[i]) * d
                Qyy = Qyy - (C1 - C2 / 3 + C2 * CY[i] * CY[i]) * d
                Qxy = Qxy - C2 * CX[i] * CY[i] * d
        else:
            mx, my = _grad(self._mu(rho), walls)
            rx, ry = _grad(rho, walls)
            Fx, Fy = fx - rho * mx, -rho * my
        if walls:
            self._fill(f, -0.5 * Fx)
        m = torch.tensordot(self.M, f, 1)
        ux, uy = (m[3] + 0.5 * Fx) / rho, (m[5] + 0.5 * Fy) / rho
        uu, uF = ux * ux + uy * uy, ux * Fx + uy * Fy
        X = [rho * (ux * ux - uy * uy), rho * ux * uy]
        if self.model == PP:
            eq = [rho * (3 * uu - 2), rho * (1 - 3 * uu)]
            src = [6 * uF, -6 * uF, 2 * (ux * Fx - uy * Fy), ux * Fy + uy * Fx]
        else:
            eq = [rho * (3 * uu - 4), rho * (4 - 3 * uu)]
            s = 6 * uF + 4 * (ux * rx + uy * ry)
            Gx, Gy = Fx + rx / 3, Fy + ry / 3
            src = [s, -s, 2 * (ux * Gx - uy * Gy), ux * Gy + uy * Gx]
            if self.A:
                # velocities of the neighbours; S = grad u + (grad u)^T
                (xx, xy), (yx, yy) = _grad(ux, False), _grad(uy, False)
                eq = [eq[0] + 2 * self.A * rho * (xx + yy), eq[1] - 2 * self.A * rho * (xx + yy)]
                X = [X[0] + 2 * self.A * rho * (xx - yy) / 3, X[1] + self.A * rho * (xy + yx) / 3]
        tr = L + 1.5 * (Qxx + Qyy)
        re, rz, rq, rn = 1 / self.te, 1 / self.tz, 1 / self.tq, 1 / self.tn
        dm = torch.stack([torch.zeros_like(rho),
                          -re * (m[1] - eq[0] - tr) + (1 - re / 2) * src[0],
                          -rz * (m[2] - eq[1] + tr) + (1 - rz / 2) * src[1],
                          Fx, -rq * (m[4] + rho * ux) - (1 - rq / 2) * Fx,
                          Fy, -rq * (m[6] + rho * uy) - (1 - rq / 2) * Fy,
                          -rn * (m[7] - X[0] + (Qxx - Qyy)) + (1 - rn / 2) * src[2],
                          -rn * (m[8] - X[1] + Qxy) + (1 - rn / 2) * src[3]])
        self.rho, self.F = rho, (Fx, Fy)
        return f + torch.tensordot(self.Mi, dm, 1)

    def stream(self, s):
        return torch.stack([torch.roll(s[i], (CY[i], CX[i]), (-2, -1)) for i in range(9)])

    def run(self, rho, steps):
        """Populations after ``steps`` steps, at the cells they left (as the framework stores them)."""
        f = self.init(rho)
        for _ in range(steps):
            s = self.collide(f)
            f = self.stream(s)
        return s


def _exact_step(case, seed):
    rho = _density(case, seed)
    if case["precision"] == 32:
        rho = rho.float().double()
    ref = _Reference(case["model"], case["Tr"] * _critical_RT(A_EOS, B_EOS), case["tau"], walls=case["walls"],
                     drive=case["drive"], split=case["nx"] // 2, A=case["A"], fx=_body(case))
    return ref.run(rho, case["steps"])


def _exact_sweep(case, seed):
    RTc, sweep = _critical_RT(A_EOS, B_EOS), _sweep(case, seed)
    out = {k: np.full(len(sweep), math.nan) for k in OBSERVABLES}
    column = lambda ids, f: torch.tensor([f(sweep[i]) for i in ids], dtype=torch.float64, device=_device())[:, None, None]  # noqa: E731
    for shape in sorted({(e["ny"], e["nx"]) for e in sweep}):  # lattices of one shape side by side
        ids = [i for i, e in enumerate(sweep) if (e["ny"], e["nx"]) == shape]
        ref = _Reference(PP, column(ids, lambda e: e["Tr"] * RTc), column(ids, lambda e: e["tau"]),
                         kappa_P=column(ids, lambda e: e["kappa_P"]))
        f = ref.init(torch.stack([torch.from_numpy(sweep[i]["rho"]) for i in ids]).to(_device()))
        for step in range(max(sweep[i]["nsteps"] for i in ids) + 1):
            s = ref.collide(f)
            for k, i in enumerate(ids):
                if sweep[i]["nsteps"] == step:
                    _observe(ref, f, k, sweep[i]["geometry"], i, out)
            f = ref.stream(s)
    return out


def _observe(ref, f, k, geometry, i, out):
    """Observables of lattice k of the batch whose state f ``ref`` has just collided, into out[.][i]."""
    rho = ref.rho[k]
    ny, nx = rho.shape
    m = torch.tensordot(ref.M, f[:, k], 1)
    u2 = ((m[3] + 0.5 * ref.F[0][k]) ** 2 + (m[5] + 0.5 * ref.F[1][k]) ** 2) / rho ** 2
    if geometry == 0:
        rl, rv, row = rho[:, nx // 2 - 1:nx // 2 + 1].mean(), rho[:, [0, nx - 1]].mean(), rho[0]
    else:
        ends = [0, 1, 2, 3, -4, -3, -2, -1]
        rl, rv = rho[ny // 2 - 2:ny // 2 + 2, nx // 2 - 2:nx // 2 + 2].mean(), rho[ends][:, ends].mean()
        row = rho[ny // 2]
    slope = (torch.roll(row, -1) - torch.roll(row, 1)).abs().max() / 2
    mass, p = rho.sum(), ref._pressure(torch.stack([rl, rv])[None, None])
    p = p.reshape(-1, 2)[k if p.numel() > 2 else 0]
    values = (rl, rv, (rl - rv) / slope, p[0] - p[1], u2.max().sqrt(), mass)
    for name, v in zip(OBSERVABLES, values):
        out[name][i] = float(v)
    if geometry == 1:
        out["radius"][i] = math.sqrt(float((mass - rv * nx * ny) / (math.pi * (rl - rv))))


def _layers(theta):
    o, out = 0, []
    for i, j in zip(DIMS, DIMS[1:]):
        out.append((theta[o:o + i * j].view(j, i), theta[o + i * j:o + i * j + j]))
        o += i * j + j
    return out


def _forward(theta, X):
    a = X
    for l, (w, b) in enumerate(_layers(theta)):
        a = a @ w.T + b
        if l < 3:
            a = 0.5 * a * (1 + torch.erf(a / math.sqrt(2.0)))
    return a


def _exact_train(case, seed):
    theta, _ = _network(seed)
    X, Y = _parameter_sets(case["sets"], seed + 1)
    t = lambda a: torch.as_tensor(np.asarray(a, dtype=np.float64), device=_device())  # noqa: E731
    st = t(lbm.Surrogate.standardisation(X, Y))
    x = (t(X) - st[0:4]) / st[4:8]
    y = t(Y)
    y[:, 1] = torch.log(y[:, 1])
    y = (y - st[8:12]) / st[12:16]
    ok = torch.isfinite(y)
    y = torch.where(ok, y, 0.0)
    p = t(theta).requires_grad_()
    m1, m2 = torch.zeros_like(p), torch.zeros_like(p)
    for it in range(case["iterations"]):
        loss = (torch.where(ok, _forward(p, x) - y, 0.0) ** 2).sum() / ok.sum()
        g, = torch.autograd.grad(loss, p)
        frac = it / (case["iterations"] - 1) if case["iterations"] > 1 else 0.0
        lr = LR / 100 + 0.5 * (LR - LR / 100) * (1 + math.cos(math.pi * frac))
        m1, m2 = 0.9 * m1 + 0.1 * g, 0.999 * m2 + 0.001 * g * g
        c1, c2 = 1 - 0.9 ** (it + 1), 1 - 0.999 ** (it + 1)
        p = (p - lr * (m1 / c1) / (torch.sqrt(m2 / c2) + 1e-8)).detach().requires_grad_()
    return {"loss": np.float64(loss.item()), "params": p.detach()}


def _exact_query(case, seed):
    theta, stats = _network(seed)
    X, _ = _parameter_sets(case["queries"], seed + 1)
    t = lambda a: torch.as_tensor(np.asarray(a, dtype=np.float64), device=_device())  # noqa: E731
    st = t(stats)
    y = _forward(t(theta), (t(X) - st[0:4]) / st[4:8]) * st[12:16] + st[8:12]
    y[:, 1] = torch.exp(y[:, 1])
    return y


def exact(case, seed):
    return dict(step=_exact_step, sweep=_exact_sweep, train=_exact_train, query=_exact_query)[case["kind"]](case, seed)
