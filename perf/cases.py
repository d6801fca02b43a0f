"""The work that a user of this library has it do, as cases to be measured.

Three families, each through the package's public entry points:

lattice   a run of one lattice: initialise from device fields, a number of
          steps, the moments back into device tensors (or, for the diagnostics
          case, the global FP64 diagnostics of a running lattice)
batch     a sweep of quasi-1-D shock tubes in one launch: initialise from
          moment blocks, run every tube, moment blocks back
net       the surrogate network: a forward pass over ragged tubes, or one
          training step (loss, gradients, Adam)

Fields that an FP32-arithmetic lattice computes are handed on as 32-bit
tensors, those of an FP64 lattice as 64-bit ones.
"""
import math
import random

import numpy as np
import torch

import paper_2201_05280_gb300 as rpk

GAMMA = 1.4
DELTA = (5.0 - 3.0 * GAMMA) / (GAMMA - 1.0)
THETA0 = 0.2948964908710633
CS = math.sqrt(GAMMA * THETA0)
KEYS = ("rho", "u", "T", "R", "Erot")


# ---------------------------------------------------------------------------
# the cases

def listed():
    return [
        # the quasi-1-D diatomic shock tube of the FP64 plain method (2000 cells,
        # reservoirs, Pr 0.71, eta_B/eta 0.6, Kn 1e-3): tiny steps, all latency
        dict(name="tube_f64", kind="lattice", nx=2000, ny=1, nz=1, precision="f64", bc="reservoir",
             rot="conservative", flow="tube", steps=100, kn=1e-3, lam=0.6, pr=0.71),
        # a small periodic box as in parity and parameter studies: latency and launches
        dict(name="box32_f32", kind="lattice", nx=32, ny=32, nz=32, precision="f32", bc="periodic",
             rot="conservative", flow="waves", steps=50, nu=0.02, lam=0.6, pr=0.71),
        # the benchmark's 256^3 decaying wave field, FP32
        dict(name="waves256_f32", kind="lattice", nx=256, ny=256, nz=256, precision="f32", bc="periodic",
             rot="conservative", flow="waves", steps=20, nu=0.02, lam=0.6, pr=0.71),
        # Taylor-Green vortex at Ma 0.3 in the paper's theta_R solver with FP16
        # deviation storage, at the relaxation times of the 512^3 run
        dict(name="tgv320_f16", kind="lattice", nx=320, ny=320, nz=320, precision="f16dev", bc="periodic",
             rot="paper", flow="tgv", steps=10, nu=9.8e-3, lam=0.6, pr=0.71),
        # an odd, ragged box with BF16 deviation storage
        dict(name="ragged_bf16", kind="lattice", nx=161, ny=127, nz=93, precision="bf16dev", bc="periodic",
             rot="conservative", flow="waves", steps=20, nu=0.04, lam=0.9, pr=0.71),
        # startup Couette flow between diffuse walls on the paper's 128 x 64 x 8 grid
        dict(name="couette_f32", kind="lattice", nx=128, ny=64, nz=8, precision="f32", bc="walls",
             rot="conservative", flow="couette", steps=50, nu=0.1, lam=0.6, pr=0.71),
        # an FP64 box, as the precision studies run it
        dict(name="box96_f64", kind="lattice", nx=96, ny=96, nz=96, precision="f64", bc="periodic",
             rot="conservative", flow="waves", steps=10, nu=0.05, lam=0.6, pr=0.71),
        # the FP64 conservation and H diagnostics of a running 256^3 FP32 lattice
        dict(name="diag256_f32", kind="diag", nx=256, ny=256, nz=256, precision="f32", bc="periodic",
             rot="conservative", flow="waves", steps=2, nu=0.02, lam=0.6, pr=0.71),
        # a parameter sweep of shock tubes with the paper's sub-stepped diffusion
        dict(name="sweep_ftcs", kind="batch", ntubes=304, lo=500, hi=1500, kn_lo=1e-3, kn_hi=1e-1,
             diffusion="ftcs"),
        # the surrogate's evaluation sweep (512 tubes of 500 to 4000 cells), backward Euler
        dict(name="sweep_implicit", kind="batch", ntubes=512, lo=500, hi=4000, kn_lo=1e-3, kn_hi=1e-1,
             diffusion="implicit"),
        # one window of a surrogate rollout: the network over all padded tubes
        dict(name="net_forward", kind="net", ntubes=512, lo=500, hi=4000, blocks=6),
        # one training step of the surrogate: 32 crops of 1024 points
        dict(name="net_train", kind="train", batch=32, crop=1024, blocks=6),
    ]


def _loguniform(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(["lattice", "lattice", "lattice", "lattice", "diag", "batch", "net", "train"])
    if kind in ("lattice", "diag"):
        form = rng.choice(["tube", "box", "box", "box", "couette"]) if kind == "lattice" else "box"
        if form == "tube":
            return dict(kind="lattice", nx=int(_loguniform(rng, 100, 4000)), ny=1, nz=1,
                        precision=rng.choice(["f64", "f32"]), bc="reservoir", rot="conservative",
                        flow="tube", steps=rng.randint(20, 100), kn=_loguniform(rng, 1e-3, 1e-2),
                        lam=rng.uniform(0.4, 2.0), pr=0.71)
        if form == "couette":
            return dict(kind="lattice", nx=rng.randint(8, 160), ny=rng.randint(8, 96), nz=rng.randint(1, 16),
                        precision=rng.choice(["f32", "f32", "f64"]), bc="walls", rot="conservative",
                        flow="couette", steps=rng.randint(10, 50), nu=rng.uniform(0.05, 0.2), lam=0.6, pr=0.71)
        precision = rng.choice(["f32", "f32", "f16dev", "bf16dev", "f64"])
        edge = _loguniform(rng, 12, 96 if precision == "f64" else 230)
        nx, ny, nz = (max(4, int(edge * rng.uniform(0.8, 1.1))) for _ in range(3))
        if rng.random() < 0.5:  # sizes as users mostly choose them
            nx = max(8, nx // 8 * 8)
        rot = rng.choice(["conservative", "conservative", "paper"])
        return dict(kind=kind, nx=nx, ny=ny, nz=nz, precision=precision, bc="periodic", rot=rot,
                    flow="waves", steps=rng.randint(5, 20), nu=rng.uniform(0.02, 0.08), lam=0.6, pr=0.71)
    if kind == "batch":
        diffusion = rng.choice(["ftcs", "implicit"])
        hi = rng.randint(600, 1500 if diffusion == "ftcs" else 4000)
        return dict(kind="batch", ntubes=int(_loguniform(rng, 40, 300 if diffusion == "ftcs" else 500)),
                    lo=rng.randint(200, 500), hi=hi, kn_lo=1e-3, kn_hi=_loguniform(rng, 1e-2, 1e-1),
                    diffusion=diffusion)
    if kind == "net":
        return dict(kind="net", ntubes=int(_loguniform(rng, 4, 500)), lo=rng.randint(100, 500),
                    hi=rng.randint(600, 4000), blocks=rng.randint(2, 6))
    return dict(kind="train", batch=rng.randint(4, 32), crop=4 * rng.randint(64, 256), blocks=rng.randint(2, 6))


# ---------------------------------------------------------------------------
# inputs

def _relax(nu, lam, pr):
    """Relaxation parameters (b = 0) of the gas with kinematic viscosity nu,
    eta_B/eta = lam and Prandtl number pr at rho = 1, theta = theta0."""
    p0, eta = THETA0, nu
    c = 2.0 * DELTA / (3.0 * (3.0 + DELTA))
    tau1 = lam * eta / (c * p0)
    tau = (eta / p0) / (1.0 - eta / (p0 * tau1))
    B = 1.0 + tau / tau1
    kappa = eta * 0.5 * (5.0 + DELTA) / pr
    k_r = kappa * 2.0 * B / (5.0 * p0 * tau) - 1.0
    return dict(delta=DELTA, tau=tau, tau1=tau1, b=0.0, k_r=k_r)


def _nsub(r, theta_max, ndim, wall=False):
    """Stable count of explicit diffusion sub-steps."""
    B = 1.0 + r["tau"] / r["tau1"]
    D = 5.0 * r["k_r"] * r["tau"] * 1.3 * theta_max / (r["delta"] * B)
    return max(1, math.ceil((2.0 * ndim + (4.0 if wall else 0.0)) * D / 0.9))


def _setup(case):
    """Relaxation parameters (with nsub) of a lattice case."""
    nu = case["kn"] * CS * case["nx"] if "kn" in case else case["nu"]
    r = _relax(nu, case["lam"], case["pr"])
    ndim = sum(case[k] > 1 for k in ("nx", "ny", "nz"))
    r["nsub"] = _nsub(r, 1.35 * THETA0, ndim, case["bc"] == "walls")
    return r


def _coords(case, dev):
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    s = torch.arange(2, device=dev, dtype=torch.float64).view(2, 1, 1, 1) * 0.5
    ar = lambda n, shape: torch.arange(n, device=dev, dtype=torch.float64).view(shape)  # noqa: E731
    return ar(nx, (1, 1, 1, nx)) + s, ar(ny, (1, 1, ny, 1)) + s, ar(nz, (1, nz, 1, 1)) + s


def _fields(case, seed, dev):
    """rho, u, T, R of a lattice case as (2, nz, ny, nx) float64 tensors, and
    the boundary states."""
    rng = random.Random(seed)
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    shape = (2, nz, ny, nx)
    X = _coords(case, dev)
    one = torch.ones(shape, device=dev, dtype=torch.float64)
    rho, T, u, edge = one.clone(), THETA0 * one, [0 * one, 0 * one, 0 * one], None
    if case["flow"] == "tube":
        # left and right state on a moderate pressure ratio, diaphragm mid way
        ratio, dens = rng.uniform(1.8, 2.2), rng.uniform(1.4, 1.6)
        left = (X[0] < 0.5 * nx).expand(shape)
        rho = torch.where(left, one, one / dens)
        T = torch.where(left, T, T * dens / ratio)
        edge = [1.0, 0, 0, 0, THETA0, THETA0, 1.0 / dens, 0, 0, 0, THETA0 * dens / ratio, THETA0 * dens / ratio]
    elif case["flow"] == "tgv":
        u0 = 0.3 * CS * rng.uniform(0.9, 1.0)
        k = [2.0 * math.pi / n for n in (nx, ny, nz)]
        ph = [rng.uniform(0, 2 * math.pi) for _ in range(3)]
        x, y, z = (k[a] * X[a] + ph[a] for a in range(3))
        u[0] = u0 * torch.sin(x) * torch.cos(y) * torch.cos(z) * one
        u[1] = -u0 * torch.cos(x) * torch.sin(y) * torch.cos(z) * one
        rho = 1.0 + u0 * u0 / (16.0 * THETA0) * (torch.cos(2 * x) + torch.cos(2 * y)) * (torch.cos(2 * z) + 2.0)
    else:
        amp = 1e-3 if case["flow"] == "couette" else 5e-3
        for c in range(3):  # a mean flow, so that the momentum is not round-off
            u[c] += 0.02 * rng.uniform(0.5, 1.0) if case["flow"] == "waves" else 0.0
        for _ in range(8 if case["flow"] == "waves" else 2):
            n = [rng.randint(-3, 3) for _ in range(3)]
            if case["flow"] == "couette":
                n[1] = 0
            arg = sum(2.0 * math.pi * n[a] / (nx, ny, nz)[a] * X[a] for a in range(3))
            ph = [rng.uniform(0, 2 * math.pi) for _ in range(5)]
            a = [amp * rng.uniform(0.5, 1.0) for _ in range(5)]
            rho += a[0] * torch.cos(arg + ph[0])
            T += THETA0 * a[1] * torch.cos(arg + ph[1])
            for c in range(3):
                u[c] += a[2 + c] * torch.cos(arg + ph[2 + c])
        if case["flow"] == "couette":
            edge = [0.0, 0.0, 0.0, THETA0, 0.1 * CS * rng.uniform(0.8, 1.0), 0.0, 0.0, 1.02 * THETA0]
    R = T * (1.0 + 0.003 * torch.cos(2 * math.pi * X[0] / nx)) if case["flow"] == "waves" else T.clone()
    return rho, torch.stack(u), T, R, edge


def _tubes(case, seed):
    """The sweep's tubes (lengths, gas, reservoirs, steps, states)."""
    rng = np.random.default_rng(seed)
    shape = np.random.default_rng(20220113)  # lengths and gases: the same work for every seed
    tubes = []
    for _ in range(case["ntubes"]):
        nx = int(shape.integers(case["lo"], case["hi"] + 1))
        kn = math.exp(shape.uniform(math.log(case["kn_lo"]), math.log(case["kn_hi"])))
        lam = float(shape.uniform(0.3, 2.0))
        ratio = float(rng.uniform(2.0, 20.0))
        r = _relax(kn * CS * nx, lam, 0.71)
        r["nsub"] = _nsub(r, THETA0, 1)
        rr, Tr = ratio ** (-1.0 / GAMMA), THETA0 * ratio ** (1.0 / GAMMA - 1.0)
        res = [1.0, 0, 0, 0, THETA0, THETA0, rr, 0, 0, 0, Tr, Tr]
        tubes.append(dict(nx=nx, nsteps=int(round(0.35 * nx / CS)), relax=r, res=res))
    return tubes


def _tube_blocks(tubes):
    """Moment blocks [4][2 nx] (rho, u_x, theta_T, E_R) of the initial states."""
    parts = []
    for t in tubes:
        nx, res = t["nx"], t["res"]
        x = np.concatenate([np.arange(nx), np.arange(nx) + 0.5])
        left = x < 0.5 * nx
        rho, T = np.where(left, res[0], res[6]), np.where(left, res[4], res[10])
        parts.append(np.stack([rho, 0 * rho, T, 0.5 * DELTA * rho * T]).astype(np.float32))
    return parts


def _net_lens(case):
    shape = np.random.default_rng(20220113)
    nx = shape.integers(case["lo"], case["hi"] + 1, size=case["ntubes"])
    return [int((2 * n + 256 + 3) // 4 * 4) for n in nx]


def _net_inputs(n, seed, dev):
    """Smooth features over n points, as packed tubes give: waves plus a little noise, 11 channels."""
    g = torch.Generator(device=dev).manual_seed(int(seed))
    k = torch.rand((11, 4), generator=g, device=dev) * 0.05
    p = torch.rand((11, 4), generator=g, device=dev) * 6.28
    pos = torch.arange(n, device=dev, dtype=torch.float32)
    x = torch.stack([torch.sin(k[c, 0] * pos + p[c, 0]) + 0.5 * torch.sin(k[c, 1] * pos + p[c, 1]) for c in range(11)], 1)
    return (x + 0.02 * torch.randn(x.shape, generator=g, device=dev)).contiguous()


def _net_params(case, seed):
    """The network's parameter vector: per layer W[o][t][i], then the biases."""
    rng = np.random.default_rng(seed)
    parts = []
    for co, taps, ci in _layers(case):
        parts.append(rng.normal(0.0, math.sqrt(1.0 / (taps * ci)), co * taps * ci))
        parts.append(rng.normal(0.0, 0.02, co))
    return np.concatenate(parts).astype(np.float32)


def _layers(case):
    return [(128, 1, 44)] + [(128, 5, 128)] * (2 * case["blocks"]) + [(16, 1, 128)]


def prepare(case, seed):
    dev = torch.device("cuda")
    kind = case["kind"]
    if kind in ("lattice", "diag"):
        rho, u, T, R, edge = _fields(case, seed, dev)
        lat = rpk.Lattice(case["nx"], case["ny"], case["nz"], precision=case["precision"],
                          bc_x="reservoir" if case["bc"] == "reservoir" else "periodic")
        lat.set_relax(**_setup(case)).set_rot_mode(case["rot"])
        if case["bc"] == "reservoir":
            lat.set_reservoirs(edge)
        if case["bc"] == "walls":
            lat.set_walls(edge[:4], edge[4:])
        n = lat.npts
        f = [rho.reshape(n).contiguous(), u.reshape(3, n).contiguous(), T.reshape(n).contiguous(), R.reshape(n).contiguous()]
        torch.cuda.synchronize()
        if kind == "diag":
            lat.init_fields(*f).step(case["steps"])
            return {"kind": kind, "lat": lat}
        out = {k: torch.empty((3, n) if k == "u" else n, device=dev, dtype=torch.float64) for k in KEYS}
        return {"kind": kind, "lat": lat, "fields": f, "steps": case["steps"], "out": out,
                "dtype": torch.float64 if case["precision"] == "f64" else torch.float32}
    if kind == "batch":
        tubes = _tubes(case, seed)
        blocks = torch.from_numpy(np.concatenate([p.ravel() for p in _tube_blocks(tubes)])).to(dev)
        bt = rpk.Batch(tubes, precision="f32", save_every=32).set_diffusion(case["diffusion"])
        bt.init_device(blocks)
        bt.autotune()
        return {"kind": kind, "batch": bt, "blocks": blocks, "out": torch.empty_like(blocks)}
    net = rpk.Net(11, 4, 128, case["blocks"], seed=0)
    net.set_params(_net_params(case, seed))
    if kind == "net":
        lens = _net_lens(case)
        x = _net_inputs(sum(lens), seed, dev)
        return {"kind": kind, "net": net, "x": x, "lens": lens, "y": torch.empty((sum(lens), 4), device=dev)}
    x, t, m = _train_data(case, seed, dev)
    return {"kind": kind, "net": net, "x": x, "t": t, "m": m}


def _train_data(case, seed, dev):
    n, L = case["batch"], case["crop"]
    x = _net_inputs(n * L, seed, dev).view(n, L, 11)
    t = (0.5 * x[:, :, :4] + 0.3 * torch.roll(x[:, :, 4:8], 3, 1)).contiguous()
    m = torch.ones((n, L), device=dev)
    edge = min(16 * case["blocks"], L // 4)
    m[:, :edge] = 0.0
    m[:, L - edge:] = 0.0
    return x, t, m


# ---------------------------------------------------------------------------
# one pass

def run(state):
    kind = state["kind"]
    if kind == "lattice":
        lat = state["lat"]
        lat.init_fields(*state["fields"])
        lat.step(state["steps"])
        m = lat.read_moments(out=state["out"])
        return [m[k].to(state["dtype"]) for k in KEYS]
    if kind == "diag":
        d = state["lat"].diagnostics()
        return [d["M"], d["J"], d["E"], d["H1"], d["min_g"]]
    if kind == "batch":
        bt = state["batch"]
        bt.init_device(state["blocks"])
        bt.run()
        return bt.moments_device(state["out"])
    net = state["net"]
    if kind == "net":
        return net.forward_ragged(state["x"], state["lens"], state["y"])
    loss = net.loss_grad(state["x"], state["t"], state["m"])
    net.adam(1e-4)
    return [loss, net.params(grads=True)]


def work(case):
    """Populations read and written once a step with the fields that carry over
    (E_R, two velocities), inputs and outputs once; the method's operations."""
    kind = case["kind"]
    if kind in ("lattice", "diag"):
        n = 2 * case["nx"] * case["ny"] * case["nz"]
        S = {"f64": 8, "f32": 4, "f16dev": 2, "bf16dev": 2}[case["precision"]]
        Rl = 8 if case["precision"] == "f64" else 4
        if kind == "diag":
            return {"bytes": n * (41 * S + Rl), "flops": n * 800.0}
        step = 82 * S + 12 * Rl
        flops = 700.0 + 25.0 * _setup(case)["nsub"]
        return {"bytes": n * (48 + 41 * S + case["steps"] * step + 41 * S + 64), "flops": n * case["steps"] * flops}
    if kind == "batch":
        by = fl = 0.0
        for t in _tubes(case, 0):
            pts, st = 2 * t["nx"], t["nsteps"]
            snaps = (st + 31) // 32
            by += pts * (st * 82 * 4 + 32 + snaps * 16)
            fl += pts * st * (700.0 + (9.0 * t["relax"]["nsub"] if case["diffusion"] == "ftcs" else 30.0))
        return {"bytes": by, "flops": fl}
    weights = sum(co * taps * ci for co, taps, ci in _layers(case))
    if kind == "net":
        pts = sum(_net_lens(case))
        return {"bytes": pts * 4 * 15 + 4 * weights, "flops": 2.0 * weights * pts / 4}
    pts = case["batch"] * case["crop"]
    return {"bytes": pts * 4 * 16 + 28 * weights, "flops": 6.0 * weights * pts / 4}


# ---------------------------------------------------------------------------
# the same in 64 bits, in plain torch

def exact(case, seed):
    dev = torch.device("cuda")
    kind = case["kind"]
    if kind in ("net", "train"):
        return _exact_net(case, seed, dev)
    if kind == "batch":
        if case["diffusion"] == "ftcs":
            return None  # up to hundreds of thousands of sub-steps one after the other
        tubes = _tubes(case, 0)
        if len(tubes) * max(t["nx"] for t in tubes) * max(t["nsteps"] for t in tubes) > 1.5e9:
            return None  # about a minute
        return _exact_batch(case, seed, dev)
    rho, u, T, R, edge = _fields(case, seed, dev)
    r = _setup(case)
    M = _Model(r, dev, rot=case["rot"])
    if case["bc"] == "reservoir":
        M.reservoirs(edge, case["nx"])
    if case["bc"] == "walls":
        M.walls(edge)
    M.init(rho, u, T, R)
    del rho, u, T, R
    for _ in range(case["steps"]):
        M.step()
    if kind == "diag":
        return M.diag()
    m = M.moments()
    n = 2 * case["nx"] * case["ny"] * case["nz"]
    return [m[0].reshape(n), m[1].reshape(3, n)] + [v.reshape(n) for v in m[2:]]


def _velocities():
    t = THETA0
    ax, out = range(3), []
    out.append(((0, 0, 0), (52 - 323 * t + 921 * t ** 2 - 1036 * t ** 3) / 52))
    for n, w in ((2, t * (12 - 38 * t + 63 * t ** 2) / 39), (4, t * (3 - 29 * t + 84 * t ** 2) / 312)):
        out += [(tuple(s * n * (b == a) for b in ax), w) for a in ax for s in (1, -1)]
    w = t * (45 * t - 6 - 77 * t ** 2) / 26
    for a in ax:
        for b in range(a + 1, 3):
            out += [(tuple(2 * (s if c == a else q if c == b else 0) for c in ax), w) for s in (1, -1) for q in (1, -1)]
    for n, w in ((2, t * (20 - 163 * t + 378 * t ** 2) / 312), (1, 8 * t * (4 - 17 * t + 21 * t ** 2) / 39)):
        out += [((n * a, n * b, n * c), w) for a in (1, -1) for b in (1, -1) for c in (1, -1)]
    return out


PAIRS = [(0, 0), (1, 1), (2, 2), (0, 1), (0, 2), (1, 2)]


class _Model:
    """The step in 64 bits on fields (2, nz, ny, nx), velocity by velocity. Relaxation parameters are numbers,
    or (1, 1, B, 1) tensors where the y axis counts independent tubes (batch=True)."""

    def __init__(self, r, dev, rot="conservative", batch=False):
        self.V = _velocities()
        self.dev, self.paper, self.batch = dev, rot == "paper", batch
        self.tau, self.tau1, self.k_r, self.nsub = r["tau"], r["tau1"], r["k_r"], r["nsub"]
        self.ts = 1.0 / (1.0 / self.tau + 1.0 / self.tau1)
        self.B = 1.0 + self.tau / self.tau1
        self.res = self.wall = None
        self.X = 1.5 / (self.tau1 * (3.0 + DELTA))

    def reservoirs(self, edge, nx):
        """States (rho, u, T, R) beyond both x ends; nx: a number, or one per tube."""
        self.res, self.nx = [edge[:6], edge[6:]], nx

    def walls(self, edge):
        self.wall = [edge[:4], edge[4:]]

    def target(self, q, rho, j, Dl):
        """f_q / w_q of a Gaussian (third-order Hermite), Dl = Lambda - theta0 I as 6 components."""
        c = [v / 2.0 for v in self.V[q][0]]
        t = THETA0
        u = [v / rho for v in j]
        cu = sum(c[a] * u[a] for a in range(3))
        uu = sum(u[a] * u[a] for a in range(3))
        cDc = sum((1 if a == b else 2) * c[a] * c[b] * Dl[k] for k, (a, b) in enumerate(PAIRS) if c[a] * c[b] != 0) if any(c) else 0.0
        tr = Dl[0] + Dl[1] + Dl[2]
        Du = [Dl[0] * u[0] + Dl[3] * u[1] + Dl[4] * u[2], Dl[3] * u[0] + Dl[1] * u[1] + Dl[5] * u[2],
              Dl[4] * u[0] + Dl[5] * u[1] + Dl[2] * u[2]]
        cDu = sum(c[a] * Du[a] for a in range(3))
        h2 = (cu * cu - t * uu) + (cDc - t * tr)
        # A3 : (ccc - t (dc + dc + dc)), A3 = uuu + D u + D u + D u
        h3 = cu ** 3 + 3.0 * cDc * cu - 3.0 * t * (uu * cu + tr * cu + 2.0 * cDu)
        return rho * (1.0 + cu / t + h2 / (2.0 * t * t) + h3 / (6.0 * t ** 3))

    def init(self, rho, u, T, R):
        self.G = torch.empty((2, len(self.V)) + tuple(rho.shape[1:]), device=self.dev, dtype=torch.float64)
        self._point(rho, u, T, R, self.G)
        th = (3.0 * T + DELTA * R) / (3.0 + DELTA)
        self.e = R.clone() if self.paper else 0.5 * DELTA * rho * (R - 0.5 / self.tau1 * (th - R))
        self.uprev = u.clone()
        self.streamed = True
        if self.res is not None:
            self.ghost = []
            for st in self.res:
                s = [v if torch.is_tensor(v) else torch.tensor(float(v), device=self.dev, dtype=torch.float64) for v in st]
                th = (3.0 * s[4] + DELTA * s[5]) / (3.0 + DELTA)
                g = [self._pointq(q, s[0], s[1:4], s[4], s[5]) for q in range(len(self.V))]
                self.ghost.append(dict(g=g, u=s[1:4], R=s[5], e=s[5] if self.paper else 0.5 * DELTA * s[0] * (s[5] - 0.5 / self.tau1 * (th - s[5])),
                                       k=2.5 * self.k_r * self.tau / self.B * s[0] * th, rho=s[0]))

    def _pointq(self, q, rho, u, T, R):
        th = (3.0 * T + DELTA * R) / (3.0 + DELTA)
        j = [rho * v for v in u]
        z = 0.0 * T
        f = self.target(q, rho, j, [T - THETA0] * 3 + [z] * 3)
        e = self.target(q, rho, j, [th - THETA0] * 3 + [z] * 3)
        return self.V[q][1] * (f - 0.5 / self.tau1 * (e - f))

    def _point(self, rho, u, T, R, G):
        for q in range(len(self.V)):
            G[:, q] = self._pointq(q, rho, u, T, R)

    def _shift(self, v, s):
        """Index shift per axis (x, y, z) of the pull of sublattice s: dst[i] = src[i - d]."""
        if v[0] & 1 == 0:
            return [c // 2 for c in v], s
        return ([1 if c > 0 else 0 for c in v] if s == 0 else [0 if c > 0 else -1 for c in v]), 1 - s

    def stream(self):
        if self.streamed:
            return self.G
        n = self.G.shape[2:]
        out = torch.empty_like(self.G)
        wall = self._wall_rho() if self.wall is not None else None
        x = torch.arange(n[2], device=self.dev).view(1, 1, -1)
        for s in range(2):
            for q, (v, w) in enumerate(self.V):
                d, src = self._shift(v, s)
                a = self.G[src, q]
                sh = [(d[0], 2)] + ([] if self.batch else [(d[1], 1), (d[2], 0)])
                sh = [(k, ax) for k, ax in sh if k and n[ax] > 1 or k and ax == 2]
                a = torch.roll(a, [k for k, _ in sh], [ax for _, ax in sh]) if sh else a
                if self.res is not None and d[0] != 0:
                    side = 0 if d[0] > 0 else 1
                    bad = (x - d[0] < 0) if side == 0 else (x - d[0] >= self.nx)
                    a = torch.where(bad, self.ghost[side]["g"][q].reshape(self.ghost[side]["g"][q].shape[-3:] if self.batch else ()), a)
                if wall is not None and d[1] != 0:
                    side = 0 if d[1] > 0 else 1
                    a = a.clone()
                    rows = slice(0, d[1]) if side == 0 else slice(n[1] + d[1], n[1])
                    a[:, rows, :] = (wall[side][0] * wall[side][1][q]).unsqueeze(1)
                out[s, q] = a
        return out

    def _wall_rho(self):
        """Per wall: the (z, x) density with which it emits what left through it, and its unit populations."""
        ny = self.G.shape[3]
        got = []
        for side in range(2):
            wl = [torch.tensor(float(v), device=self.dev, dtype=torch.float64) for v in self.wall[side]]
            unit = [self._pointq(q, torch.ones_like(wl[3]), wl[:3], wl[3], wl[3]) for q in range(len(self.V))]
            mass, emit = 0.0, 0.0
            for s in range(2):
                for q, (v, w) in enumerate(self.V):
                    d, _ = self._shift(v, s)
                    if d[1] != 0 and (d[1] > 0) == (side == 0):
                        emit = emit + abs(d[1]) * unit[q]
                    # where population q of sublattice s goes along y
                    go = v[1] // 2 if v[0] & 1 == 0 else (0 if v[1] > 0 else -1) if s == 0 else (1 if v[1] > 0 else 0)
                    if go < 0 and side == 0:
                        mass = mass + self.G[s, q][:, :-go, :].sum(1)
                    if go > 0 and side == 1:
                        mass = mass + self.G[s, q][:, ny - go:, :].sum(1)
            got.append((mass / emit, unit))
        return got

    def recover(self, G):
        rho = G.sum(1)
        j = [sum(G[:, q] * (v[a] / 2.0) for q, (v, w) in enumerate(self.V) if v[a]) for a in range(3)]
        P = [sum(G[:, q] * (v[a] * v[b] / 4.0) for q, (v, w) in enumerate(self.V) if v[a] * v[b]) for a, b in PAIRS]
        u = [v / rho for v in j]
        Tg = (P[0] + P[1] + P[2] - rho * (u[0] ** 2 + u[1] ** 2 + u[2] ** 2)) / (3.0 * rho)
        a_ = DELTA * self.X / 3.0
        if self.paper:
            R = self.e
            T = (Tg + a_ * R) / (1.0 + a_)
        else:
            Rt = 2.0 * self.e / (DELTA * rho)
            det = (1.0 + a_) * (1.0 + self.X) - a_ * self.X
            T = (Tg * (1.0 + self.X) + a_ * Rt) / det
            R = ((1.0 + a_) * Rt + self.X * Tg) / det
        return rho, j, u, P, Tg, T, R

    def _mix(self, m):
        """Lambda - theta0 I of the mixed target (b = 0) and theta."""
        rho, j, u, P, Tg, T, R = m
        th = (3.0 * T + DELTA * R) / (3.0 + DELTA)
        iso = self.ts / self.tau * T + self.ts / self.tau1 * th - THETA0
        z = torch.zeros_like(iso)
        return [iso, iso, iso, z, z, z], th

    def step(self):
        G = self.stream()
        m = self.recover(G)
        rho, j, u, P, Tg, T, R = m
        Dl, th = self._mix(m)
        beta = 1.0 / (2.0 * self.ts + 1.0)
        for q, (v, w) in enumerate(self.V):
            G[:, q] = (1.0 - 2.0 * beta) * G[:, q] + 2.0 * beta * w * self.target(q, rho, j, Dl)
        kap = 2.5 * self.k_r * self.tau / self.B * rho * th
        u = torch.stack(u)
        if self.paper:
            keep, mixt = 1.0 / (1.0 + self.X), self.X / (1.0 + self.X)
            r = keep * R + mixt * T
            rp = r - sum(u[a] * (self._nb(r, a, 1) - r) for a in self._axes(r))
            rc = 0.5 * (r + rp - sum(u[a] * (rp - self._nb(rp, a, -1)) for a in self._axes(r)))
            for _ in range(self.nsub):
                lap = sum(self._nb(rc, a, 1) - 2.0 * rc + self._nb(rc, a, -1) for a in self._axes(r))
                rc = rc + 2.0 * kap / (rho * DELTA * self.nsub) * lap
            e = keep * rc + mixt * T
        else:
            e = self._transport(self.e + 0.5 * DELTA * rho * (th - R) / self.tau1, rho, kap, 1.5 * u - 0.5 * self.uprev)
        self.G, self.e, self.uprev, self.streamed = G, e, u, False

    def _axes(self, a):
        return [0] if self.batch else [k for k in range(3) if a.shape[3 - k] > 1]

    def _nb(self, a, axis, d, low=None, high=None):
        """a at the neighbour i + d along the axis; low / high stand beyond the reservoirs or walls."""
        out = torch.roll(a, -d, 3 - axis)
        edge = (axis == 0 and self.res is not None) or (axis == 1 and self.wall is not None)
        if edge and low is not None:
            n = a.shape[3 - axis]
            i = torch.arange(n, device=self.dev).view([-1 if k == 3 - axis else 1 for k in range(4)])
            last = self.nx if axis == 0 else n
            out = torch.where(i + d < 0, low, out) if d < 0 else torch.where(i + d >= last, high, out)
        return out

    def _transport(self, e, rho, kap, v):
        g = self.ghost if self.res is not None else None
        zero = torch.zeros_like(e)

        def ends(axis, key):
            if axis == 0 and g is not None:
                return g[0][key], g[1][key]
            return zero, zero  # a wall: no flux through it

        def flux(f, axis, d):
            lo, hi = ends(axis, "e")
            if axis == 0 and g is not None:
                lo, hi = lo * g[0]["u"][0], hi * g[1]["u"][0]
            return self._nb(f * v[axis], axis, d, lo, hi)

        ep = e - sum(flux(e, a, 1) - e * v[a] for a in self._axes(e))
        e = 0.5 * (e + ep - sum(ep * v[a] - flux(ep, a, -1) for a in self._axes(e)))
        if self.nsub == "implicit":
            return self._implicit(e, rho, kap)
        low, high = (torch.tensor(v, device=self.dev, dtype=torch.float64).view(2, 1, 1, 1) for v in ([3.0, 1.0 / 3.0], [1.0 / 3.0, 3.0]))
        for _ in range(self.nsub):
            th = 2.0 * e / (DELTA * rho)
            acc = zero
            for a in self._axes(e):
                for d in (1, -1):
                    tl = th_ = kl = kh = None
                    if a == 0 and g is not None:
                        tl, th_, kl, kh = (g[0]["R"], g[1]["R"], g[0]["k"], g[1]["k"])
                    if a == 1 and self.wall is not None:
                        wl, wh = self.wall[0][3], self.wall[1][3]
                        tl = wl + (wl - th) * low
                        th_ = wh + (wh - th) * high
                        kl = kh = kap
                    acc = acc + 0.5 * (kap + self._nb(kap, a, d, kl, kh)) * (self._nb(th, a, d, tl, th_) - th)
            e = e + acc / self.nsub
        return e

    def _implicit(self, e, rho, kap):
        """Backward Euler along x between the reservoirs: parallel cyclic reduction."""
        g = self.ghost
        n = e.shape[3]
        x = torch.arange(n, device=self.dev).view(1, 1, 1, -1)
        km = 0.5 * (kap + self._nb(kap, 0, -1, g[0]["k"], g[1]["k"]))
        kp = 0.5 * (kap + self._nb(kap, 0, 1, g[0]["k"], g[1]["k"]))
        b = 0.5 * DELTA * rho + km + kp
        d = e + torch.where(x == 0, km * g[0]["R"], 0.0) + torch.where(x == self.nx - 1, kp * g[1]["R"], 0.0)
        a, c = torch.where(x == 0, 0.0, -km), torch.where(x >= self.nx - 1, 0.0, -kp)
        inside = x < self.nx
        a, c, d, b = (torch.where(inside, t, f) for t, f in ((a, 0.0), (c, 0.0), (d, 0.0), (b, 1.0)))
        pad = torch.nn.functional.pad
        h = 1
        while h < n:
            lo = lambda t, f: pad(t[..., :-h], (h, 0), value=f)  # noqa: E731, B023
            hi = lambda t, f: pad(t[..., h:], (0, h), value=f)  # noqa: E731, B023
            al, ga = -a / lo(b, 1.0), -c / hi(b, 1.0)
            b, d = b + al * lo(c, 0.0) + ga * hi(a, 0.0), d + al * lo(d, 0.0) + ga * hi(d, 0.0)
            a, c = al * lo(a, 0.0), ga * hi(c, 0.0)
            h *= 2
        return 0.5 * DELTA * rho * d / b

    def moments(self):
        rho, j, u, P, Tg, T, R = self.recover(self.stream())
        return rho, torch.stack(u), T, R, 0.5 * DELTA * rho * R

    def diag(self):
        G = self.stream()
        m = self.recover(G)
        rho, j, u, P, Tg, T, R = m
        Dl, _ = self._mix(m)
        er = 0.5 * DELTA * rho * R if self.paper else self.e
        M, J, E = float(rho.sum()), np.array([float(v.sum()) for v in j]), float((0.5 * (P[0] + P[1] + P[2]) + er).sum())
        beta = 1.0 / (2.0 * self.ts + 1.0)
        H = float((-0.5 * DELTA * rho * torch.log(R)).sum())
        for q, (v, w) in enumerate(self.V):
            f = (1.0 - beta) * G[:, q] + beta * w * self.target(q, rho, j, Dl)
            H += float((f * torch.log(f / w) - f).sum())
        return [M, J, E, H, float(G.min())]


def _exact_batch(case, seed, dev):
    tubes = _tubes(case, seed)
    B, X = len(tubes), max(t["nx"] for t in tubes)
    col = lambda f: torch.tensor([float(f(t)) for t in tubes], device=dev, dtype=torch.float64).view(1, 1, B, 1)  # noqa: E731
    r = {k: col(lambda t, k=k: t["relax"][k]) for k in ("tau", "tau1", "k_r")}
    r["nsub"] = "implicit"
    M = _Model(r, dev, batch=True)
    nx = torch.tensor([t["nx"] for t in tubes], device=dev).view(1, B, 1)
    M.reservoirs([col(lambda t, k=k: t["res"][k]) for k in range(12)], nx)
    f = torch.ones((4, 2, 1, B, X), dtype=torch.float64)
    f[1], f[2], f[3] = 0.0, THETA0, 0.5 * DELTA * THETA0
    for i, (t, p) in enumerate(zip(tubes, _tube_blocks(tubes))):
        f[:, :, 0, i, :t["nx"]] = torch.from_numpy(p.astype(np.float64)).view(4, 2, t["nx"])
    f = f.to(dev)
    rho, T, R = f[0], f[2], 2.0 * f[3] / (DELTA * f[0])
    M.init(rho, torch.stack([f[1], 0 * f[1], 0 * f[1]]), T, R)
    steps = torch.tensor([t["nsteps"] for t in tubes], device=dev).view(1, 1, B, 1)
    out = None
    order = sorted({t["nsteps"] for t in tubes})
    done = 0
    for last in order:
        while done < last:
            M.step()
            done += 1
        m = M.moments()
        got = torch.stack([m[0], m[1][0], m[2], m[4]])
        out = got if out is None else torch.where(steps >= last, got, out)
    return torch.cat([out[:, :, 0, i, :t["nx"]].reshape(-1) for i, t in enumerate(tubes)])


def _exact_net(case, seed, dev):
    p = torch.from_numpy(_net_params(case, seed).astype(np.float64)).to(dev).requires_grad_(case["kind"] == "train")
    W, at = [], 0
    for co, taps, ci in _layers(case):
        n = co * taps * ci
        W.append((p[at:at + n].view(co, taps, ci), p[at + n:at + n + co]))
        at += n + co

    def conv(x, layer):  # x (sequences, positions, channels), zero beyond the ends
        w, b = layer
        r = w.shape[1] // 2
        n = x.shape[1]
        xp = torch.nn.functional.pad(x, (0, 0, r, r))
        return sum(xp[:, t:t + n] @ w[:, t].T for t in range(w.shape[1])) + b

    def net(x):
        s, n, _ = x.shape
        h = conv(x.reshape(s, n // 4, 44), W[0])
        for i in range(case["blocks"]):
            h = h + conv(torch.relu(conv(torch.relu(h), W[1 + 2 * i])), W[2 + 2 * i])
        return conv(torch.relu(h), W[-1]).reshape(s, n, 4)

    if case["kind"] == "net":
        lens = _net_lens(case)
        x = _net_inputs(sum(lens), seed, dev).double()
        with torch.no_grad():
            return torch.cat([net(t[None])[0] for t in x.split(lens)])
    x, t, m = (v.double() for v in _train_data(case, seed, dev))
    loss = (m[..., None] * (net(x) - t) ** 2).sum() / (m.sum() * 4)
    loss.backward()
    return [float(loss), p.grad.cpu().numpy()]
