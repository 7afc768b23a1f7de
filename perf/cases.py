"""Performance cases: what users of this framework have it do, each as one
whole pass through the public Python entry points.

A pass sets the initial state, advances it and reads the result out, as a
program that studies one configuration after another does; the lattice, batch
or network object (its buffers, launch plans, autotuned schedule) is made once
in prepare() and kept.  Sizes are those of the repository's configurations,
tests and bench (inputs.py, the paper's validation grids, bench.py) or lie
between them.
"""
import math

import numpy as np
import torch

import paper_2010_01847_gb300 as plbm
from paper_2010_01847_gb300 import warmstart

ISO, FLUX, DIFF = plbm.ISOTHERMAL, plbm.HEAT_FLUX, plbm.DIFFUSE

# The D2Q8 velocities and weights of the paper (Eqs. 14, 17, 18) for exact().
CX = (1, 0, -1, 0, 1, -1, -1, 1)
CY = (0, 1, 0, -1, 1, 1, -1, -1)
WEIGHT = (2 / 9,) * 4 + (1 / 36,) * 4
HFLUX = (1 / 3,) * 4 + (1 / 12,) * 4


def listed():
    return [
        # the smallest calls: the paper's thin film between two isothermal
        # sides (ragged rows), looked at every 100 steps
        dict(name="film_301x3", kind="film", nx=301, ny=3, precision="fp32", steps=100, windows=1),
        # the Poiseuille channel of the paper at its usual resolution, run in
        # residual windows towards its steady state
        dict(name="channel_128x32", kind="channel", nx=128, ny=32, precision="fp32", steps=500,
             windows=2),
        # the paper's square with three isothermal sides and one heated side
        # (odd sizes, sides on both axes)
        dict(name="square_201x201", kind="square", nx=201, ny=201, precision="fp32", steps=500,
             windows=1),
        # one wide channel of the batched study's range, on its own
        dict(name="channel_1024x256", kind="channel", nx=1024, ny=256, precision="fp32",
             steps=200, windows=2),
        # the reference precision, for end states and error studies
        dict(name="channel_512x128_fp64", kind="channel", nx=512, ny=128, precision="fp64",
             steps=200, windows=1),
        # decaying heat mode with noise, a lattice about the size of the L2
        dict(name="heat_2048x2048", kind="heat", nx=2048, ny=2048, precision="fp32", steps=200,
             windows=1),
        # the headline workload, one residual window
        dict(name="heat_8192x8192", kind="heat", nx=8192, ny=8192, precision="fp32", steps=100,
             windows=1),
        # 16-bit storage: FP16 rounded to nearest on a large lattice ...
        dict(name="heat_4096x4096_fp16", kind="heat", nx=4096, ny=4096, precision="fp16",
             steps=100, windows=1),
        # ... and BF16 with stochastic rounding, as long runs use it
        dict(name="heat_2048x2048_bf16", kind="heat", nx=2048, ny=2048, precision="bf16",
             rounding="stochastic", steps=100, windows=1),
        # uneven channels advanced together from the analytic start, two
        # check windows of the steady-state solve
        dict(name="batch_48", kind="batch", count=48, wmax=512, steps=150, windows=2),
        # three-dimensional heat mode
        dict(name="d3q14_192", kind="d3q14", nx=192, ny=192, nz=192, precision="fp32",
             steps=300, windows=1),
        # training and prediction of the warm-start network
        dict(name="mlp_train_512", kind="mlp", n=1024, batch=512, steps=100, predict=512),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("film", "channel", "channel", "channel", "square", "heat", "heat", "heat",
                       "heat16", "heat16", "batch", "d3q14", "mlp"))
    if kind == "film":          # the paper's films and plates: 3 rows, odd lengths
        return dict(kind="film", nx=_log(rng, 21, 801), ny=rng.randint(3, 5),
                    precision=rng.choice(("fp32", "fp32", "fp64")), steps=2 * rng.randint(25, 150),
                    windows=1)
    if kind == "channel":       # widths of the batched study, length 4 W (or thereabouts)
        w = _log(rng, 16, 512)
        nx = 4 * w + rng.choice((0, 0, 0, -3, 2))
        return dict(kind="channel", nx=nx, ny=w,
                    precision="fp64" if w <= 200 and rng.random() < 0.25 else "fp32",
                    steps=2 * rng.randint(25, 150), windows=rng.randint(1, 2))
    if kind == "square":
        n = _log(rng, 21, 401)
        return dict(kind="square", nx=n, ny=n + rng.randint(-5, 5), precision="fp32",
                    steps=2 * rng.randint(50, 250), windows=1)
    if kind == "heat":
        nx, ny = _log(rng, 64, 8192), _log(rng, 64, 4096)
        nx = nx // 16 * 16 + rng.choice((0, 0, 0, 0, 4, 6, 9))
        return dict(kind="heat", nx=nx, ny=ny, precision="fp32", steps=2 * rng.randint(25, 60),
                    windows=1)
    if kind == "heat16":
        nx, ny = _log(rng, 256, 4096) // 8 * 8, _log(rng, 256, 4096)
        return dict(kind="heat", nx=nx, ny=ny, precision=rng.choice(("fp16", "bf16")),
                    rounding=rng.choice(("nearest", "stochastic")), steps=2 * rng.randint(20, 50),
                    windows=1)
    if kind == "batch":
        return dict(kind="batch", count=rng.randint(6, 48), wmax=_log(rng, 64, 512),
                    steps=2 * rng.randint(25, 75), windows=2)
    if kind == "d3q14":
        n = _log(rng, 24, 176)
        return dict(kind="d3q14", nx=n + rng.randint(0, 16), ny=n + rng.randint(-5, 5), nz=n,
                    precision=rng.choice(("fp32", "fp32", "fp32", "fp64")) if n <= 96 else "fp32",
                    steps=rng.randint(50, 200), windows=1)
    return dict(kind="mlp", n=_log(rng, 256, 4096), batch=rng.choice((128, 256, 512, 512, 1000)),
                steps=rng.randint(30, 100), predict=_log(rng, 8, 1024))


# ---------------------------------------------------------------------------
# The physical setting of a case (relaxation times in lattice units by Eq. 48,
# boundaries) and its seeded initial fields, shared by prepare() and exact().
def _tau(kn, length):
    return kn * length * math.sqrt(3.0 / 5.0)


def _setting(case, seed):
    rng = np.random.default_rng([seed, 17])
    kind, nx, ny = case["kind"], case["nx"], case["ny"]
    kn_n, kn_r = 10 ** rng.uniform(-1.5, -1.0), 10 ** rng.uniform(-0.5, 0.5)
    sides, bc_x, bc_y, delta_e = None, plbm.PERIODIC, plbm.PERIODIC, 0.0
    if kind == "channel":
        length, bc_x, bc_y, delta_e = max(ny - 1, 24), plbm.PERIODIC_GRADIENT, plbm.DIFFUSE_WALLS, 1e-3
    elif kind == "film":
        length, bc_x = max(nx - 1, 24), plbm.SIDES
        sides = [(ISO, 1.0005), (ISO, 0.9995), (None, 0), (None, 0)]
    elif kind == "square":
        length, bc_x, bc_y = max(nx - 1, 24), plbm.SIDES, plbm.SIDES
        sides = [(ISO, 1.0), (ISO, 1.0), (ISO, 1.0), (FLUX, 1e-4)]
    else:
        length, kn_n, kn_r = 512.0, 0.01 * 10 ** rng.uniform(-0.1, 0.3), 0.1 * 10 ** rng.uniform(-0.3, 0.3)
    return _tau(kn_n, length), _tau(kn_r, length), bc_x, bc_y, delta_e, sides


def _start(case, seed, shape, device="cuda"):
    """e = 1 + a sine mode with a seeded phase (oblique where there are rows
    enough, along x in films) + U[-1e-6, 1e-6) noise."""
    g = torch.Generator(device=device)
    g.manual_seed(int(seed) * 2 + 1)
    nx = shape[-1]
    x = torch.arange(nx, dtype=torch.float64, device=device)
    mode = max(1, round(nx / 512))
    phase = 0.1 * (int(seed) % 61)
    e = torch.rand(shape, generator=g, dtype=torch.float64, device=device)
    e.mul_(2e-6).sub_(1e-6)
    arg = 2.0 * math.pi * mode * x / nx + phase
    if shape[-2] >= 16:
        y = torch.arange(shape[-2], dtype=torch.float64, device=device)
        arg = arg[None, :] + (2.0 * math.pi * max(1, round(shape[-2] / 512)) / shape[-2] * y)[:, None]
    e += 1.0 + 1e-3 * torch.sin(arg)
    return e


def _channels(case, seed=0):
    """Channels of widths 16..wmax, length 4 W, as the batched study draws
    them: the widths belong to the case, the Knudsen numbers to the seed (kept
    inside the scheme's stable range, tau >= 0.6)."""
    widths = np.random.default_rng([case["count"], case["wmax"]]).integers(16, case["wmax"] + 1,
                                                                         case["count"])
    rng = np.random.default_rng([seed, 23])
    out = []
    for w in map(int, widths):
        while True:
            tau_n = _tau(10 ** rng.uniform(-3, -1), w - 1)
            tau_r = _tau(10 ** rng.uniform(-1, 1), w - 1)
            if 1.0 / (1.0 / tau_n + 1.0 / tau_r) >= 0.1:
                break
        out.append(dict(nx=4 * w, ny=w, tau_N=tau_n, tau_R=tau_r, bc_x=plbm.PERIODIC_GRADIENT,
                        bc_y=plbm.DIFFUSE_WALLS, delta_e=1e-3))
    return out


def _net_data(case, seed):
    """Network inputs in [-1, 1]^3 and smooth 512-point targets of the size
    of the profile corrections the warm start learns; seeded weights."""
    rng = np.random.default_rng([seed, 29])
    n = case["n"]
    x = rng.uniform(-1, 1, (n, 3))
    j = np.arange(512) / 255.0
    t = sum(0.1 * (1 + 0.5 * x[:, a:a + 1]) * np.sin((a + 1) * j[None, :] * 3 + 2 * x[:, (a + 1) % 3][:, None])
            for a in range(3))
    params = []
    for k, m in zip(warmstart.WIDTHS[:-1], warmstart.WIDTHS[1:]):
        a = math.sqrt(6.0 / (k + m))
        params += [rng.uniform(-a, a, m * k), np.zeros(m)]
    xp = rng.uniform(-1, 1, (case["predict"], 3))
    return (x.astype(np.float32), t.astype(np.float32), np.concatenate(params).astype(np.float32),
            xp.astype(np.float32))


LR, LR_FINAL, NET_SEED = 1e-3, 1e-5, 7


def prepare(case, seed):
    kind = case["kind"]
    if kind == "mlp":
        x, t, p, xp = _net_data(case, seed)
        net = plbm.Mlp(warmstart.WIDTHS, max_batch=max(case["batch"], case["predict"]))
        return dict(case=case, net=net, x=torch.from_numpy(x).cuda(), t=torch.from_numpy(t).cuda(),
                    p=p, xp=torch.from_numpy(xp).cuda())
    if kind == "batch":
        ch = _channels(case, seed)
        start = plbm.analytic_profiles(ch)
        b = plbm.Batch(ch)
        b.init_profiles(start)
        b.autotune(10)
        return dict(case=case, batch=b, start=start)
    tau_n, tau_r, *bc, sides = _setting(case, seed) if kind != "d3q14" else \
        (*_setting(dict(case, kind="heat"), seed)[:2], None)
    if kind == "d3q14":
        shape = (case["nz"], case["ny"], case["nx"])
        lat = plbm.LatticeND(plbm.D3Q14, shape, tau_n, tau_r, precision=case["precision"])
        return dict(case=case, lat=lat, e=_start(case, seed, shape).cpu().numpy())
    lat = plbm.Lattice(case["nx"], case["ny"], tau_n, tau_r, bc[0], bc[1], bc[2],
                       precision=case["precision"], sides=sides,
                       rounding=case.get("rounding", "nearest"))
    e = _start(case, seed, (case["ny"], case["nx"]))
    return dict(case=case, lat=lat, e=e, qx=0.01 * (e - 1.0), qy=torch.zeros_like(e))


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "mlp":
        net = state["net"]
        net.set_params(state["p"])
        loss = net.train(state["x"], state["t"], case["steps"], case["batch"], LR, LR_FINAL,
                         seed=NET_SEED)
        return dict(loss=loss, y=net.forward(state["xp"]), params=net.params())
    if kind == "batch":
        b = state["batch"]
        b.init_profiles(state["start"])
        steps, r = b.solve(1e-8, case["steps"], case["steps"] * case["windows"])
        return dict(steps=steps, r=r, profiles=b.profiles())
    lat = state["lat"]
    if kind == "d3q14":
        lat.init(state["e"])
        lat.step(case["steps"])
        e, q = lat.moments()
        return dict(e=e, q=q)
    lat.init(state["e"], state["qx"], state["qy"])
    if kind in ("film", "square"):            # a fixed time, then the fields
        lat.step(case["steps"])
        return _fields(lat)
    r = []
    for _ in range(case["windows"]):          # residual windows
        r.append(lat.step_residual(case["steps"]))
    return dict(r=[v[0] for v in r], energy=[v[1] for v in r], **_fields(lat))


def _fields(lat):
    e = torch.empty((lat.ny, lat.nx), dtype=torch.float64, device="cuda")
    q = torch.empty((2, lat.ny, lat.nx), dtype=torch.float64, device="cuda")
    lat.moments_device(out=(e, q[0], q[1]))
    return dict(e=e, q=q)


def work(case):
    """Inputs read once, outputs written once, and the arithmetic of the
    collision: 65 operations per node and step in two dimensions (15 for the
    moments, 10 for the flux, 5 for each of 8 relaxations), 107 on D3Q14."""
    kind = case["kind"]
    if kind == "mlp":
        pairs = list(zip(warmstart.WIDTHS[:-1], warmstart.WIDTHS[1:]))
        weights = sum(k * m for k, m in pairs)
        params = weights + sum(warmstart.WIDTHS[1:])
        macs = case["batch"] * (3 * weights - pairs[0][0] * pairs[0][1])
        return dict(bytes=4.0 * (2 * params + case["n"] * 515 + case["predict"] * 515),
                    flops=2.0 * macs * case["steps"] + 2.0 * weights * case["predict"])
    n_steps = case["steps"] * case["windows"]
    if kind == "batch":
        nodes = float(sum(c["nx"] * c["ny"] for c in _channels(case)))
        # the populations of so many channels cannot stay on the chip: one
        # read and write of the state per window
        return dict(bytes=nodes * 64.0 * case["windows"] + case["count"] * 4096.0,
                    flops=65.0 * nodes * n_steps)
    if kind == "d3q14":
        nodes = float(case["nx"] * case["ny"] * case["nz"])
        return dict(bytes=nodes * 40.0, flops=107.0 * nodes * n_steps)
    nodes = float(case["nx"] * case["ny"])
    return dict(bytes=nodes * 48.0, flops=65.0 * nodes * n_steps)


# ---------------------------------------------------------------------------
# The method in 64 bits with plain torch: push as rolls, on deviations from
# the rest equilibrium at e = 1.
def _step2d(f, tau_n, tau_r, bc_x, bc_y, delta_e, sides, n):
    """n steps of the state f (deviations, [8] of [ny, nx])."""
    tau = 1.0 / (1.0 / tau_n + 1.0 / tau_r) + 0.5
    kappa = 2.0 * tau_r / (2.0 * tau_r + 1.0)
    sigma = (1.0 - 0.5 / tau) / tau_r
    ny, nx = f[0].shape
    for _ in range(n):
        rho = sum(f)
        qx = (f[0] - f[2] + f[4] - f[6] + f[7] - f[5]) * kappa
        qy = (f[1] - f[3] + f[4] - f[6] + f[5] - f[7]) * kappa
        g = []
        for i in range(8):
            t = HFLUX[i] * (CX[i] * qx + CY[i] * qy)
            p = f[i] - (f[i] - WEIGHT[i] * rho - t) / tau - sigma * t
            p = torch.roll(p, (CY[i], CX[i]), (0, 1))
            if bc_x == plbm.PERIODIC_GRADIENT and CX[i] > 0:
                p[:, 0] += WEIGHT[i] * delta_e
            if bc_x == plbm.PERIODIC_GRADIENT and CX[i] < 0:
                p[:, nx - 1] -= WEIGHT[i] * delta_e
            g.append(p)
        f = g
        # Section 2.5: unknown populations of each bounded side from the incident ones
        todo = []
        if bc_y == plbm.DIFFUSE_WALLS:
            todo = [(2, DIFF, 0.0), (3, DIFF, 0.0)]
        if sides:
            for s in (2, 3, 0, 1):
                if sides[s][0] is not None:
                    todo.append((s, *sides[s]))
        at = {0: (slice(None), 0), 1: (slice(None), nx - 1), 2: (0, slice(None)), 3: (ny - 1, slice(None))}
        into = {0: lambda i: CX[i] > 0, 1: lambda i: CX[i] < 0, 2: lambda i: CY[i] > 0, 3: lambda i: CY[i] < 0}
        out = {0: lambda i: CX[i] < 0, 1: lambda i: CX[i] > 0, 2: lambda i: CY[i] < 0, 3: lambda i: CY[i] > 0}
        for s, kind, value in todo:
            if kind == ISO:
                continue
            inc = sum(f[i][at[s]] for i in range(8) if out[s](i)) + (value / kappa if kind == FLUX else 0.0)
            for i in range(8):
                if into[s](i):
                    f[i][at[s]] = WEIGHT[i] / (5.0 / 18.0) * inc
        for s, kind, value in sorted(todo, reverse=True):       # left last: it wins a corner
            if kind == ISO:
                for i in range(8):
                    f[i][at[s]] = WEIGHT[i] * (value - 1.0)
    return f


def _equilibrium2d(e, qx, qy):
    return [WEIGHT[i] * (e - 1.0) + HFLUX[i] * (CX[i] * qx + CY[i] * qy) for i in range(8)]


def _moments2d(f, tau_r):
    kappa = 2.0 * tau_r / (2.0 * tau_r + 1.0)
    return dict(e=1.0 + sum(f), q=torch.stack([(f[0] - f[2] + f[4] - f[6] + f[7] - f[5]) * kappa,
                                               (f[1] - f[3] + f[4] - f[6] + f[5] - f[7]) * kappa]))


def _exact3d(case, seed):
    tau_n, tau_r = _setting(dict(case, kind="heat"), seed)[:2]
    tau = 1.0 / (1.0 / tau_n + 1.0 / tau_r) + 0.5
    kappa = 2.0 * tau_r / (2.0 * tau_r + 1.0)
    sigma = (1.0 - 0.5 / tau) / tau_r
    c = [(1, 0, 0), (0, 1, 0), (0, 0, 1), (1, 1, 1), (1, 1, -1), (1, -1, 1), (1, -1, -1)]
    c = c + [tuple(-v for v in b) for b in c]
    w = [1 / 9 if sum(map(abs, b)) == 1 else 1 / 24 for b in c]
    h = [1 / 3 if sum(map(abs, b)) == 1 else 1 / 24 for b in c]
    e = _start(case, seed, (case["nz"], case["ny"], case["nx"]))
    f = [w[i] * (e - 1.0) for i in range(14)]

    def moments(f):
        q = []
        for a in range(3):
            m = 0
            for i in range(14):
                if c[i][a]:
                    m = m + c[i][a] * f[i]
            q.append(m * kappa)
        return sum(f), q

    for _ in range(case["steps"]):
        rho, q = moments(f)
        for i in range(14):
            t = h[i] * sum(c[i][a] * q[a] for a in range(3) if c[i][a])
            p = f[i] - (f[i] - w[i] * rho - t) / tau - sigma * t
            f[i] = torch.roll(p, (c[i][2], c[i][1], c[i][0]), (0, 1, 2))
    rho, q = moments(f)
    return dict(e=1.0 + rho, q=torch.stack(q))


def _eq68(ch):
    """The analytic flux profile (Eq. 68) at 256 points across the channel."""
    tau_c, d = 1.0 / (1.0 / ch["tau_N"] + 1.0 / ch["tau_R"]), ch["ny"] - 1.0
    kn_eff = math.sqrt(tau_c * ch["tau_R"] / 3.0) / d
    kn_c = math.sqrt(5.0 / 3.0) * tau_c / d
    y = np.arange(256) / 255.0
    a = math.exp(-1.0 / kn_eff)
    return 1.0 - (np.exp((y - 1.0) / kn_eff) + np.exp(-y / kn_eff)) / \
        (1.0 + a + (8.0 / 15.0) * (kn_c / kn_eff) * (1.0 - a))


def _exact_batch(case, seed):
    n = case["steps"] * case["windows"]
    prof = []
    for ch in _channels(case, seed):
        nx, ny, de, tau_r = ch["nx"], ch["ny"], ch["delta_e"], ch["tau_R"]
        unit = 5.0 / 9.0 * tau_r * de / nx
        pts = np.float32(_eq68(ch)).astype(np.float64)
        q_row = torch.from_numpy(np.interp(np.arange(ny) / (ny - 1) * 255.0, np.arange(256), pts)).cuda()
        aff = de / nx * (torch.arange(nx, dtype=torch.float64, device="cuda") - 0.5 * (nx - 1))
        e = (1.0 - aff).repeat(ny, 1)
        qx = (q_row * unit)[:, None].repeat(1, nx)
        f = _equilibrium2d(e, qx, torch.zeros_like(e))
        f = _step2d(f, ch["tau_N"], tau_r, plbm.PERIODIC_GRADIENT, plbm.DIFFUSE_WALLS, de, None, n)
        m = _moments2d(f, tau_r)
        e, qx = m["e"], m["q"][0]
        rows = torch.stack([qx.mean(1) / unit, (e + aff - 1.0).mean(1) * nx / de]).cpu().numpy()
        yf = np.arange(256) / 255.0 * (ny - 1)
        prof.append(np.concatenate([np.interp(yf, np.arange(ny), v) for v in rows]))
    return dict(steps=None, r=None, profiles=np.stack(prof))


def _exact_mlp(case, seed):
    x, t, p, xp = _net_data(case, seed)
    x, t, xp = (torch.from_numpy(v).double().cuda() for v in (x, t, xp))
    p = torch.from_numpy(p).double().cuda().requires_grad_(True)
    m, v = torch.zeros_like(p), torch.zeros_like(p)
    n, batch, steps = case["n"], case["batch"], case["steps"]

    def net(p, x):
        o = 0
        pairs = list(zip(warmstart.WIDTHS[:-1], warmstart.WIDTHS[1:]))
        for l, (k, w) in enumerate(pairs):
            x = x @ p[o:o + k * w].view(w, k).T + p[o + k * w:o + k * w + w]
            o += k * w + w
            if l < len(pairs) - 1:
                x = torch.nn.functional.gelu(x)
        return x

    loss = []
    for s in range(steps):
        rows = np.arange(batch) % n
        if batch < n:                  # SplitMix64 of the seed and the draw's number
            with np.errstate(over="ignore"):
                z = (np.uint64(NET_SEED) ^ (np.uint64(s * batch) + np.arange(batch, dtype=np.uint64))) \
                    + np.uint64(0x9E3779B97F4A7C15)
                z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
                z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
                rows = ((z ^ (z >> np.uint64(31))) % np.uint64(n)).astype(np.int64)
        rows = torch.from_numpy(rows).cuda()
        err = (net(p, x[rows]) - t[rows]).square().mean()
        (g,) = torch.autograd.grad(err, p)
        with torch.no_grad():
            m = 0.9 * m + 0.1 * g
            v = 0.999 * v + 0.001 * g * g
            lr = LR_FINAL + 0.5 * (LR - LR_FINAL) * (1.0 + math.cos(math.pi * s / steps))
            p -= lr * (m / (1 - 0.9 ** (s + 1))) / ((v / (1 - 0.999 ** (s + 1))).sqrt() + 1e-8)
        loss.append(err.detach())
    with torch.no_grad():
        return dict(loss=torch.stack(loss), y=net(p, xp), params=p.detach())


def exact(case, seed):
    kind = case["kind"]
    if kind == "mlp":
        return _exact_mlp(case, seed)
    if kind == "batch":
        return _exact_batch(case, seed)
    if kind == "d3q14":
        return _exact3d(case, seed)
    tau_n, tau_r, bc_x, bc_y, delta_e, sides = _setting(case, seed)
    e = _start(case, seed, (case["ny"], case["nx"]))
    f = _equilibrium2d(e, 0.01 * (e - 1.0), torch.zeros_like(e))
    energy = []
    for _ in range(case["windows"]):
        f = _step2d(f, tau_n, tau_r, bc_x, bc_y, delta_e, sides, case["steps"])
        energy.append(float(f[0].numel() + sum(f).sum()))
    if kind in ("film", "square"):
        return _moments2d(f, tau_r)
    return dict(r=[None] * case["windows"], energy=energy, **_moments2d(f, tau_r))
