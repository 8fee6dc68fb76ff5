"""What is measured: the time steps, batches and surrogate training that users of this
framework run, each through its public entry points (Simulation, Batch, Mlp).

Kinds of case:
  sim     one run on one grid: `steps` time steps, then the fields (density, velocity,
          chemical potential) on the device.  `start` 1: the pass also sets the initial
          fields, as each run of a parameter study does; 0: it continues the run.
          `shift`: everything (and the walls) moves along x at that speed, a moving frame.
  batch   uneven instances advanced together, then every instance's fields on the host.
  fit     minibatch Adam steps on the surrogate network, its weights, and its prediction.
  grad    the surrogate's loss and gradient on one batch.

`exact` restates the method of arXiv:1906.09530 in 64 bits: the compact scheme of
Eqs. 37-39 by its symbol (FFT along each line), everything else node by node.
"""
import math
import random

import numpy as np
import torch

import paper_1906_09530_gb300 as P

F64 = torch.float64
# D2Q9 velocities and weights (Sec. 2)
EX = (0, 1, 0, -1, 0, 1, -1, -1, 1)
EY = (0, 0, 1, 0, -1, 1, 1, -1, -1)
WQ = (4 / 9,) + (1 / 9,) * 4 + (1 / 36,) * 4
MRT_RATES = (1.64, 1.54, 1.9)  # s_e, s_eps, s_q (Sec. 2)
NET = (4, 256, 256, 256, 256)  # the surrogate's layer widths


def sim_case(name, nx, ny, steps, **kw):
    c = dict(kind="sim", nx=nx, ny=ny, steps=steps, precision="mixed", order=6, eos="cs",
             T_r=0.5, kappa=0.1, tau=1.0, k=0.5, shape="drop", size=0.2 * min(nx, ny),
             width=8.0, collision="bgk", walls=False, shift=0.0, mu_max=0.0, cap_steps=0,
             start=0, lone=False)
    c.update(kw)
    return dict(c, name=name) if name else c


def listed():
    return [
        # the flat interface whose equilibrium and coexistence curve are run for 1e5 steps,
        # looked at every 500, seen from a moving frame: a small grid, bound by latency
        sim_case("slab-8x400", 8, 400, 500, T_r=0.8, k=0.1, shape="slab", size=200.0, width=40.0,
                 shift=0.05),
        # the FP64 drop of the accuracy tests: 4th order, k = 1
        sim_case("drop-128-fp64", 128, 128, 200, precision="fp64", T_r=0.7, k=1.0, order=4,
                 size=24.0, width=4.0),
        # an odd grid (no vector path), multiple relaxation times, 4th order
        sim_case("ragged-333x277-mrt", 333, 277, 100, T_r=0.7, k=0.3, order=4, width=13.0,
                 collision="mrt"),
        # the paper's drop splash: Peng-Robinson water, walls in y, the upper limit of the
        # chemical potential; each pass is the start of another run
        sim_case("splash-1000x300-pr", 1000, 300, 200, eos="pr", T_r=0.6, kappa=0.005, tau=0.7,
                 k=0.1, shape="splash", size=50.0, width=20.0, walls=True, mu_max=6.0,
                 cap_steps=1000, start=1),
        # one step at a time, the fields read on the device after each (a coupled program)
        sim_case("drop-1024-lone", 1024, 1024, 1, size=200.0, lone=True),
        # the headline workload, back to back
        sim_case("drop-1024", 1024, 1024, 200, size=200.0),
        # the same drop in FP64
        sim_case("drop-1024-fp64", 1024, 1024, 10, precision="fp64", size=200.0),
        # a drop at density ratio 8e4, where the density's derivatives are double-float
        sim_case("drop-1000-low-T", 1000, 1000, 50, T_r=0.35, k=0.2, size=250.0, width=20.0),
        # a grid far above the L2
        sim_case("drop-4096", 4096, 4096, 10, size=800.0),
        # many uneven drops and slabs over the whole temperature range
        dict(name="batch-24", kind="batch", n=24, pick=1234, lo=64, hi=512, odd=False, t_lo=0.3,
             t_hi=0.9, steps=200),
        # the surrogate's fit at its default minibatch, and its prediction
        dict(name="fit-256", kind="fit", batch=256, minibatches=16, lr=1e-3),
        # full-batch gradient of the surrogate's loss
        dict(name="grad-32768", kind="grad", batch=32768),
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(("sim", "sim", "sim", "sim", "fp64", "splash", "batch", "fit", "grad"))
    if kind == "fit":
        return dict(kind="fit", batch=_log_int(rng, 16, 2048), minibatches=rng.randint(4, 16),
                    lr=1e-3)
    if kind == "grad":
        return dict(kind="grad", batch=_log_int(rng, 64, 32768))
    if kind == "batch":
        return dict(kind="batch", n=rng.randint(4, 24), pick=rng.randint(0, 10**6), lo=64, hi=400,
                    odd=True, t_lo=round(rng.uniform(0.3, 0.5), 3),
                    t_hi=round(rng.uniform(0.6, 0.9), 3), steps=rng.randint(20, 100))
    if kind == "splash":
        nx, ny = _log_int(rng, 400, 2048), _log_int(rng, 300, 1024)
        return sim_case(None, nx, ny, rng.randint(20, 200), eos="pr", T_r=0.6, kappa=0.005,
                        tau=rng.choice((0.7, 1.25)), k=0.1, shape="splash", size=50.0, width=20.0,
                        walls=True, shift=rng.choice((0.0, 0.03)), mu_max=6.0, cap_steps=1000,
                        start=1)
    # FP64 grids up to 1024^2 nodes, mixed ones up to 4096^2; one in three narrow slabs
    top = 1024 if kind == "fp64" else 4096
    if rng.random() < 0.33:
        nx, ny, shape = _log_int(rng, 8, 512), rng.randint(200, 1024), "slab"
        size = ny / 2
    else:
        nx, ny, shape = _log_int(rng, 96, top), _log_int(rng, 96, top), "drop"
        size = 0.22 * min(nx, ny)
    if rng.random() < 0.4:  # grids whose rows are whole 16-byte pieces, as most users choose
        nx = max(8, nx // 8 * 8)
    T_r, k = rng.choice(((0.5, 0.5), (0.6, 0.5), (0.7, 0.3), (0.35, 0.2), (0.8, 0.1)))
    if size < 4.0 / k:  # too small for that interface's width
        T_r, k = 0.6, 0.5
    mrt = T_r == 0.7 and rng.random() < 0.5
    steps = int(min(200, max(5, 1.6e8 / (nx * ny + 2e5))))
    return sim_case(None, nx, ny, max(4, steps // 12) if kind == "fp64" else steps,
                    precision="fp64" if kind == "fp64" else "mixed", T_r=T_r, k=k,
                    order=rng.choice((4, 6, 6)), shape=shape, size=size,
                    width=min(4.0 / k, size / 2), collision="mrt" if mrt else "bgk",
                    shift=0.05 if shape == "slab" else 0.0)


# ---- inputs -----------------------------------------------------------------


def _eos(case):
    """(T, T_c, pressure, mu0, rho_max) of the case's equation of state (Sec. 3.2)."""
    if case.get("eos", "cs") == "cs":
        a, b, alpha_m, rmax = 1.0, 4.0, 0.0, 1.0

        def A(r):
            e = 0.25 * b * r
            return r * (1 + e + e * e - e**3) / (1 - e) ** 3

        def dA(r):
            e = 0.25 * b * r
            return (1 + 4 * e + 4 * e**2 - 4 * e**3 + e**4) / (1 - e) ** 4

        def B(r):
            return a * r * r

        def dB(r):
            return 2 * a * r
    else:  # Peng-Robinson, water
        a, b, w = 2 / 49, 2 / 21, 0.344
        alpha_m, rmax = 0.37464 + 1.54226 * w - 0.26992 * w * w, 21 / 2

        def A(r):
            return r / (1 - b * r)

        def dA(r):
            return 1 / (1 - b * r) ** 2

        def B(r):
            return a * r * r / (1 + 2 * b * r - (b * r) ** 2)

        def dB(r):
            return a * (2 * r + 2 * b * r * r) / (1 + 2 * b * r - (b * r) ** 2) ** 2
    # T_c: the maximum of the spinodal temperature dB/dA
    lo, hi = 1e-3 * rmax, 0.95 * rmax
    for _ in range(200):
        x, y = lo + (hi - lo) / 3, hi - (hi - lo) / 3
        lo, hi = (x, hi) if dB(x) / dA(x) < dB(y) / dA(y) else (lo, y)
    Tc = dB(0.5 * (lo + hi)) / dA(0.5 * (lo + hi))
    T = case["T_r"] * Tc
    al = (1 + alpha_m * (1 - math.sqrt(case["T_r"]))) ** 2

    def p0(r):
        return T * A(r) - al * B(r)

    def mu0(r, log=math.log):
        if alpha_m == 0.0:
            e = 0.25 * b * r
            return T * ((3 - e) / (1 - e) ** 3 + log(r) + 1) - 2 * a * r
        s2 = math.sqrt(2.0)
        return (T * log(r / (1 - b * r)) + T / (1 - b * r)
                - a * al / (2 * s2 * b) * log((s2 - 1 + b * r) / (s2 + 1 - b * r))
                - a * al * r / (1 + 2 * b * r - (b * r) ** 2))

    def dp0(r):
        return T * dA(r) - al * dB(r)

    return p0, dp0, mu0, 0.5 * (lo + hi), rmax


def _bisect(f, lo, hi):
    up = f(lo) < 0
    for _ in range(200):
        mid = 0.5 * (lo + hi)
        lo, hi = (mid, hi) if (f(mid) < 0) == up else (lo, mid)
    return 0.5 * (lo + hi)


def coexistence(case):
    """Maxwell densities (gas, liquid): equal pressure and chemical potential."""
    p0, dp0, mu0, rc, rmax = _eos(case)
    sg, sl = _bisect(dp0, 1e-12 * rc, rc), _bisect(dp0, rc, rmax * (1 - 1e-12))

    def gas(m):
        return math.exp(_bisect(lambda x: mu0(math.exp(x)) - m, -200.0, math.log(sg)))

    top = _bisect(lambda r: mu0(r) - mu0(sg), sl, rmax * (1 - 1e-12))
    rl = _bisect(lambda r: p0(r) - p0(gas(mu0(r))), sl, top)
    return gas(mu0(rl)), rl


def initial(case, seed):
    """(rho, ux, uy): tanh interfaces between the coexistence densities, the drop moved by
    up to two nodes and 1e-4 of multiplicative noise by the seed."""
    rg, rl = coexistence(case)
    nx, ny, W = case["nx"], case["ny"], case["width"]
    gen = torch.Generator(device="cuda").manual_seed(seed)
    r = torch.rand((2,), generator=gen, device="cuda", dtype=F64) * 4 - 2
    y = torch.arange(ny, device="cuda", dtype=F64)[:, None]
    x = torch.arange(nx, device="cuda", dtype=F64)[None, :]
    ux = torch.full((ny, nx), case["shift"], device="cuda", dtype=F64) if case["shift"] else None
    uy = None

    def side(d):  # 1 well inside (d < 0), 0 outside
        return 0.5 * (1.0 - torch.tanh(2.0 * d / W))

    if case["shape"] == "slab":
        phi = side((y - ny / 2 - r[0]).abs() - case["size"] / 2).expand(ny, nx)
    elif case["shape"] == "drop":
        phi = side(torch.hypot(x - nx / 2 - r[0], y - ny / 2 - r[1]) - case["size"])
    else:  # a drop falling onto the film on the bottom wall
        film, gap = 30.0, 25.0
        d = side(torch.hypot(x - nx / 2 - r[0], y - film - case["size"] - gap) - case["size"])
        phi = torch.maximum(side(y - film).expand(ny, nx), d)
        ux, uy = torch.zeros_like(d) if ux is None else ux, -0.1 * d
    eps = torch.rand((ny, nx), generator=gen, device="cuda", dtype=F64) * 2 - 1
    return (rg + (rl - rg) * phi) * (1 + 1e-4 * eps), ux, uy


def instances(case):
    """The batch's instances: square grids of uneven sides, temperatures log-spaced."""
    rng, out = random.Random(case["pick"]), []
    for i in range(case["n"]):
        side = (_log_int(rng, case["lo"], case["hi"]) if case["odd"] else
                rng.choice([s for s in (64, 128, 256, 512) if case["lo"] <= s <= case["hi"]]))
        T = case["t_lo"] * (case["t_hi"] / case["t_lo"]) ** (i / max(case["n"] - 1, 1))
        k = 0.5 if T >= 0.45 else 0.3
        slab = rng.random() < 0.5
        out.append(sim_case(None, side, side, case["steps"], T_r=T, k=k, width=4.0 / k,
                            shape="slab" if slab else "drop", shift=0.05,
                            size=0.5 * side if slab else 0.25 * side))
    return out


def net_inputs(case, seed):
    """(inputs [n][4], targets [n][256], weights): scaled inputs in [-1, 1], interface-like
    targets, Glorot weights."""
    rng = np.random.default_rng(seed)
    n = case["batch"] * case.get("minibatches", 1)
    x = rng.uniform(-1, 1, (n, 4)).astype(np.float32)
    s = np.linspace(-4, 4, 256)
    t = 0.5 + 0.5 * np.tanh(s[None, :] * (1.2 + 0.5 * x[:, :1]) + x[:, 1:2]) * (1 + 0.2 * x[:, 2:3])
    w = []
    for a, b in zip(NET[:-1], NET[1:]):
        lim = math.sqrt(6 / (a + b))
        w += [rng.uniform(-lim, lim, a * b), rng.uniform(-0.1, 0.1, b)]
    return x, t.astype(np.float32), np.concatenate(w).astype(np.float32)


# ---- the cases --------------------------------------------------------------


def prepare(case, seed):
    if case["kind"] in ("fit", "grad"):
        x, t, w = net_inputs(case, seed)
        net = P.Mlp(case["batch"])
        net.set_params(w)
        return dict(case=case, net=net, x=torch.from_numpy(x).cuda(), t=torch.from_numpy(t).cuda())
    if case["kind"] == "batch":
        inst = instances(case)
        batch = P.Batch([dict(nx=c["nx"], ny=c["ny"], T_r=c["T_r"], k=c["k"], kappa=c["kappa"])
                         for c in inst])
        for i, c in enumerate(inst):
            rho, ux, _ = initial(c, seed + 1000 * i)
            batch.set_fields(i, rho.cpu().numpy(), ux.cpu().numpy())
        return dict(case=case, batch=batch)
    eos = P.make_eos("pr", omega=0.344) if case["eos"] == "pr" else P.cs_eos()
    sim = P.Simulation(case["nx"], case["ny"], case["T_r"], case["kappa"], case["tau"], case["k"],
                       fd_order=case["order"], precision=case["precision"], eos=eos,
                       mu_max=case["mu_max"] or math.inf, mu_cap_steps=case["cap_steps"],
                       collision=case["collision"], walls_y=case["walls"],
                       wall_ux=(case["shift"] if case["walls"] else 0.0,) * 2)
    fields = initial(case, seed)
    sim.set_fields_device(*fields)
    sim.check()
    return dict(case=case, sim=sim, fields=fields if case["start"] else None)


def run(state):
    case = state["case"]
    if case["kind"] == "sim":
        sim = state["sim"]
        if state["fields"] is not None:
            sim.set_fields_device(*state["fields"])
        if case["lone"]:
            sim.step_async(case["steps"])
        else:
            sim.step(case["steps"])
        return sim.fields_device()
    if case["kind"] == "batch":
        state["batch"].step(case["steps"])
        return [np.stack(state["batch"].fields(i)) for i in range(case["n"])]
    net, x, t, n = state["net"], state["x"], state["t"], case["batch"]
    if case["kind"] == "grad":
        return net.loss_grad(x, t)
    for s in range(0, len(x), n):
        net.train_step(x[s:s + n], t[s:s + n], case["lr"])
    return net.get_params(), net.forward(x[:n])


def work(case):
    """Populations in and out (once where they fit the L2 between steps, else every step),
    the initial fields and the outputs; the network's operands."""
    if case["kind"] in ("fit", "grad"):
        n, m = case["batch"], case.get("minibatches", 1)
        w = sum(a * b for a, b in zip(NET[:-1], NET[1:]))
        par = w + sum(NET[1:])
        flops = 2.0 * n * (2 * w + w - NET[0] * NET[1])
        return dict(bytes=float(m * (n * 260 * 4 + 8 * par)), flops=m * flops)
    if case["kind"] == "batch":
        each = [work(c) for c in instances(case)]
        return {q: sum(e[q] for e in each) for q in ("bytes", "flops")}
    size = 8 if case["precision"] == "fp64" else 4
    nodes = case["nx"] * case["ny"]
    trips = 1 if 9 * size * nodes < 1e8 else case["steps"]
    fields = 32 + (24 if case["start"] else 0)
    return dict(bytes=float(nodes * (trips * 18 * size + fields)),
                flops=230.0 * nodes * case["steps"])


# ---- 64-bit values ----------------------------------------------------------


def _derivative(order, dim, n, walls):
    """The compact first derivative along `dim` (Eqs. 37-39) as a function of a field; with
    walls, of the field extended evenly (odd for a field that is itself a derivative)."""
    al = 1 / 3 if order == 6 else 1 / 4
    a, b = 2 / 3 * (al + 2), (4 * al - 1) / 3
    m = 2 * n if walls else n
    th = 2 * math.pi * torch.arange(m // 2 + 1, device="cuda", dtype=F64) / m
    sym = 1j * (a * torch.sin(th) + b / 2 * torch.sin(2 * th)) / (1 + 2 * al * torch.cos(th))
    if m % 2 == 0:
        sym[-1] = 0
    sym = sym.reshape((-1, 1) if dim == 0 else (1, -1))

    def ext(u, sign):
        return torch.cat((u, sign * u.flip(dim)), dim) if walls else u

    def D(u, sign=1):
        d = torch.fft.irfft(torch.fft.rfft(ext(u, sign), dim=dim) * sym, n=m, dim=dim)
        return d.narrow(dim, 0, n)

    return D


def _exact_sim(case, seed):
    rho, ux, uy = initial(case, seed)
    ny, nx = rho.shape
    _, _, mu0, _, rmax = _eos(case)
    k2 = case["k"] ** 2
    Dx, Dy = _derivative(case["order"], 1, nx, False), \
        _derivative(case["order"], 0, ny, case["walls"])
    t = 0

    def force(rho):
        gx, gy = Dx(rho), Dy(rho)
        lap = Dx(gx) + Dy(gy, -1)
        if case["cap_steps"] > t:  # the upper limit, which also takes nodes past the EOS pole
            m = k2 * mu0(rho.clamp(max=rmax * (1 - 1e-9)), torch.log) - case["kappa"] * lap
            m = torch.where(rho >= rmax, torch.full_like(m, math.inf), m)
            m = m.clamp(max=k2 * case["mu_max"])
        else:
            m = k2 * mu0(rho, torch.log) - case["kappa"] * lap
        return m, -rho * Dx(m) + gx / 3, -rho * Dy(m) + gy / 3

    def feq(rho, u, v):
        uu = 1.5 * (u * u + v * v)
        return [w * rho * (1 + 3 * (x * u + y * v) + 4.5 * (x * u + y * v) ** 2 - uu)
                for w, x, y in zip(WQ, EX, EY)]

    def moments(f):
        return (sum(f), sum(x * g for x, g in zip(EX, f) if x),
                sum(y * g for y, g in zip(EY, f) if y))

    relax = None
    if case["collision"] == "mrt":
        ex, ey = np.array(EX, float), np.array(EY, float)
        c = ex**2 + ey**2
        M = np.stack([np.ones(9), 3 * c - 4, 4 - 10.5 * c + 4.5 * c * c, ex, (3 * c - 5) * ex, ey,
                      (3 * c - 5) * ey, ex**2 - ey**2, ex * ey])
        se, seps, sq = MRT_RATES
        S = np.diag([0, se, seps, 0, sq, 0, sq, 1 / case["tau"], 1 / case["tau"]])
        relax = np.linalg.inv(M) @ S @ M

    zero = torch.zeros_like(rho)
    f = feq(rho, zero if ux is None else ux, zero if uy is None else uy)
    rho = sum(f)
    mu, Fx, Fy = force(rho)
    for _ in range(case["steps"]):
        r, jx, jy = moments(f)
        u, v = jx / r, jy / r
        e0, e1 = feq(r, u, v), feq(r, u + Fx / r, v + Fy / r)
        if relax is None:
            post = [g - (g - a) / case["tau"] + b - a for g, a, b in zip(f, e0, e1)]
        else:
            d = [g - a for g, a in zip(f, e0)]
            post = [g - sum(q * z for q, z in zip(row, d) if abs(q) > 1e-15) + b - a
                    for g, row, a, b in zip(f, relax, e0, e1)]
        f = [torch.roll(g, (y, x), (0, 1)) for g, x, y in zip(post, EX, EY)]
        if case["walls"]:  # halfway bounce-back, walls moving along x (Ladd)
            for row, into in ((0, ((2, 4), (5, 7), (6, 8))), (ny - 1, ((4, 2), (7, 5), (8, 6)))):
                c = sum(g[row] for g in post) * case["shift"] / 6
                for i, j in into:
                    f[i][row] = post[j][row] + EX[i] * c
        rho = sum(f)
        t += 1
        mu, Fx, Fy = force(rho)
    r, jx, jy = moments(f)
    return r, (jx + 0.5 * Fx) / r, (jy + 0.5 * Fy) / r, mu


def _exact_net(case, seed):
    x, t, p = (torch.from_numpy(v).cuda().double() for v in net_inputs(case, seed))

    def layers(p):
        o = 0
        for a, b in zip(NET[:-1], NET[1:]):
            yield p[o:o + a * b].reshape(a, b), p[o + a * b:o + a * b + b]
            o += a * b + b

    def forward(p, x):
        for i, (w, b) in enumerate(layers(p)):
            x = x @ w + b
            x = torch.tanh(x) if i < 3 else x
        return x

    def gradient(p, x, t):
        p = p.detach().requires_grad_()
        loss = ((forward(p, x) - t) ** 2).mean()
        return loss.detach(), torch.autograd.grad(loss, p)[0]

    n = case["batch"]
    if case["kind"] == "grad":
        return gradient(p, x, t)
    m, v = torch.zeros_like(p), torch.zeros_like(p)
    for i, s in enumerate(range(0, len(x), n), 1):
        g = gradient(p, x[s:s + n], t[s:s + n])[1]
        m, v = 0.9 * m + 0.1 * g, 0.999 * v + 0.001 * g * g
        p = p - case["lr"] * (m / (1 - 0.9**i)) / ((v / (1 - 0.999**i)).sqrt() + 1e-8)
    return p, forward(p, x[:n])


def exact(case, seed):
    if case["kind"] in ("fit", "grad"):
        return _exact_net(case, seed)
    if case["kind"] == "batch":
        return [torch.stack(_exact_sim(c, seed + 1000 * i)) for i, c in enumerate(instances(case))]
    return _exact_sim(case, seed)
