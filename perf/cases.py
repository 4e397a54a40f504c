"""The work that a user of the solver has it do, as cases that can be timed and
whose results can be compared: flow past bodies with the force of every step
(one domain or a batch of uneven ones), gradients of the force, step-by-step
monitoring, and a whole job from the mask to the forces.

Every case goes through the Python binding.  Inputs depend on the seed alone:
the body's incidence, a gust profile on the inlet (a different velocity in
every row), the discs of a porous medium, the perturbation of a start state.
`exact` restates a case in torch FP64 (plain array operations, no code of this
repository beyond this file).
"""
import math

import numpy as np
import torch

from paper_2210_10377_gb300 import binding

U0 = 0.05
SCHEMES = ("A", "B", "DRTT", "A_RTT", "SI")
BATCH_SCHEMES = ("B", "DRTT", "SI")
ELEM = {"f64": 8, "f32": 4, "f32dev": 4, "f16dev": 2}
FLOPS_PER_UPDATE = 130  # one BGK collision (Section II), counted on the written formula


def tau_of(chord, re):
    return 0.5 + 3.0 * U0 * chord / re


def listed():
    return [
        # a control loop: one step, one force, again (latency of single calls)
        dict(name="monitor_f32dev_512x256", kind="monitor", storage="f32dev", nx=512, ny=256, chord=64.0,
             alpha=2.0, tau=tau_of(64.0, 200.0), steps=25),
        # the FP64 reference runs of precision studies: small grid, every scheme
        dict(name="flow_f64_256x128", kind="flow", storage="f64", nx=256, ny=128, chord=32.0, alpha=0.0,
             tau=tau_of(32.0, 100.0), steps=120),
        # the differentiation grid's forward run: many steps of a grid that fits in cache
        dict(name="flow_f32dev_512x256", kind="flow", storage="f32dev", nx=512, ny=256, chord=64.0, alpha=2.0,
             tau=tau_of(64.0, 200.0), steps=1000),
        # Section VI's cylinder at an odd diameter, plain FP32 populations, ragged rows
        dict(name="flow_f32_cylinder_1500x125", kind="flow", storage="f32", nx=1500, ny=125, chord=25.0,
             body="cylinder", alpha=0.0, tau=tau_of(25.0, 100.0), steps=600),
        # a periodic porous medium driven by a body force, bodies everywhere, odd sizes
        dict(name="porous_f32dev_1001x333", kind="porous", storage="f32dev", nx=1001, ny=333, discs=60,
             radius=9.0, tau=0.8, steps=200),
        # the throughput workload: NACA0012, chord 256 at 4 degrees, Re 1000
        dict(name="flow_f32dev_4096x2048", kind="flow", storage="f32dev", nx=4096, ny=2048, chord=256.0,
             alpha=4.0, tau=tau_of(256.0, 1000.0), steps=300),
        # the precision workload: chord 512 at 6 degrees, Re 2000, FP16 deviations
        dict(name="flow_f16dev_8192x4096", kind="flow", storage="f16dev", nx=8192, ny=4096, chord=512.0,
             alpha=6.0, tau=tau_of(512.0, 2000.0), steps=400),
        # Section VI's convergence study: five cylinders, uneven domains, one batch
        dict(name="sweep_f32_cylinders", kind="sweep", storage="f32", what="cylinders", diameters="10,15,20,30,40",
             tau=0.0, steps=600),
        # a design sweep: NACA00xx sections of random thickness, chord, incidence and Re
        dict(name="sweep_f16dev_naca_12", kind="sweep", storage="f16dev", what="naca", domains=12, lo=48, hi=128,
             tau=0.0, steps=300),
        # gradient of the mean drag on the differentiation grid
        dict(name="grad_f32dev_512x256", kind="grad", storage="f32dev", nx=512, ny=256, chord=64.0, alpha=2.0,
             tau=tau_of(64.0, 200.0), steps=1000, window=250),
        # the same at the throughput size, a short horizon
        dict(name="grad_f32dev_4096x2048", kind="grad", storage="f32dev", nx=4096, ny=2048, chord=256.0, alpha=4.0,
             tau=tau_of(256.0, 1000.0), steps=64, window=16),
        # one whole job: voxelise, create, run, read forces, coefficients and the state, release
        dict(name="job_f32dev_1024x512", kind="job", storage="f32dev", nx=1024, ny=512, chord=64.0, alpha=4.0,
             tau=tau_of(64.0, 250.0), steps=250),
    ]


def draw(rng):
    def log(lo, hi):
        return math.exp(rng.uniform(math.log(lo), math.log(hi)))

    def section(nx_lo, nx_hi):
        nx = int(log(nx_lo, nx_hi))
        ny = max(48, int(nx * rng.uniform(0.3, 0.6)))
        chord = round(nx * rng.uniform(0.05, 0.12), 1)
        return dict(nx=nx, ny=ny, chord=chord, alpha=round(rng.uniform(-6.0, 6.0), 2), tau=round(0.5 + log(0.02, 0.2), 4))

    kind = rng.choices(("flow", "porous", "sweep", "grad", "monitor", "job"), (9, 2, 3, 3, 2, 1))[0]
    storage = rng.choice(("f64", "f32", "f32dev", "f32dev", "f16dev", "f16dev"))
    if kind == "flow":
        c = section(192, 8000)
        budget = log(2e7, 4e9 if storage != "f64" else 5e8)
        return dict(kind=kind, storage=storage, steps=int(min(1500, max(20, budget / (c["nx"] * c["ny"])))), **c)
    if kind == "porous":
        nx, ny = int(log(128, 1500)), int(log(96, 700))
        return dict(kind=kind, storage=storage, nx=nx, ny=ny, discs=rng.randint(8, 60), radius=round(rng.uniform(3, 10), 1),
                    tau=round(rng.uniform(0.6, 1.1), 3), steps=rng.randint(20, 300))
    if kind == "sweep":
        if rng.random() < 0.4:
            ds = sorted(rng.sample(range(8, 41), rng.randint(3, 6)))
            return dict(kind=kind, storage=storage, what="cylinders", diameters=",".join(map(str, ds)), tau=0.0,
                        steps=rng.randint(100, 600))
        return dict(kind=kind, storage=storage, what="naca", domains=rng.randint(3, 14), lo=rng.randint(24, 56),
                    hi=rng.randint(60, 128), tau=0.0, steps=rng.randint(60, 300))
    if kind == "grad":
        c = section(128, 2400)
        steps = rng.randint(24, 400)
        return dict(kind=kind, storage=storage, steps=steps, window=rng.randint(1, steps), **c)
    if kind == "monitor":
        return dict(kind=kind, storage=storage, steps=rng.randint(8, 40), **section(128, 3000))
    return dict(kind=kind, storage=storage, steps=rng.randint(40, 300), **section(192, 3000))


# ---------------------------------------------------------------- inputs


def _rng(seed):
    return np.random.Generator(np.random.PCG64(seed))


def _gust(g, ny):
    """Inlet velocity of every row: U0 with three gust harmonics of up to 2 %."""
    y = np.arange(ny) / ny
    u = np.ones(ny)
    for m in (1, 2, 3):
        u += g.uniform(0.005, 0.02) * np.sin(2.0 * np.pi * (m * y + g.uniform()))
    return U0 * u


def _section(c, seed):
    """The single-domain inputs: the section's incidence, its place and the inlet."""
    g = _rng(seed)
    alpha = c["alpha"] + g.uniform(-1.0, 1.0)
    return dict(nx=c["nx"], ny=c["ny"], chord=c["chord"], alpha=alpha, thickness=0.12, xc=0.3125 * c["nx"],
                yc=(c["ny"] - 1) / 2.0, tau=c["tau"], u=_gust(g, c["ny"]), body=c.get("body", "naca"))


def _sweep(c, seed):
    g = _rng(seed)
    if c["what"] == "cylinders":
        out = []
        for d in map(int, c["diameters"].split(",")):
            re = g.uniform(90.0, 110.0)
            out.append(dict(nx=60 * d, ny=5 * d, chord=float(d), alpha=0.0, thickness=0.0, xc=15.0 * d,
                            yc=(5 * d - 1) / 2.0, tau=tau_of(d, re), u=_gust(g, 5 * d), body="cylinder"))
        return out
    out = []
    chords = _rng(c["domains"]).uniform(c["lo"], c["hi"], c["domains"])  # the sizes are the case's, not the seed's
    for k in range(c["domains"]):
        cb = int(round(chords[k]))
        out.append(dict(nx=8 * cb, ny=4 * cb, chord=float(cb), alpha=g.uniform(-8.0, 8.0), thickness=g.uniform(0.08, 0.15),
                        xc=2.5 * cb, yc=(4 * cb - 1) / 2.0, tau=tau_of(cb, 10.0 ** g.uniform(2.0, 3.0)),
                        u=_gust(g, 4 * cb), body="naca"))
    return out


def _discs(c, seed):
    """Random discs, wrapping through all edges, and the start velocity of every row."""
    g = _rng(seed)
    nx, ny = c["nx"], c["ny"]
    mask = np.zeros((ny, nx), np.uint8)
    x, y = np.arange(nx)[None, :], np.arange(ny)[:, None]
    for _ in range(c["discs"]):
        r = g.uniform(1.0, c["radius"])
        dx = np.abs(x - g.uniform(0, nx))
        dy = np.abs(y - g.uniform(0, ny))
        mask[np.minimum(dx, nx - dx) ** 2 + np.minimum(dy, ny - dy) ** 2 <= r * r] = 1
    return mask, _gust(g, ny), (2e-6, -5e-7)


def _mask(p):
    """The body on the device, as a user voxelises it."""
    if p["body"] == "cylinder":
        return binding.cylinder_mask(p["nx"], p["ny"], p["xc"], p["yc"], p["chord"])
    return binding.naca_mask(p["nx"], p["ny"], p["chord"], p["thickness"], p["alpha"], p["xc"], p["yc"])


def _start(p, seed, device):
    """A perturbed start state: the equilibrium of the inlet velocities, each
    population times 1 + U[-1e-3, 1e-3], FP64 [9][ny][nx]."""
    u = torch.from_numpy(p["u"]).to(device)
    feq = torch.stack([W[i] * (1.0 + 3.0 * CX[i] * u + 4.5 * (CX[i] * u) ** 2 - 1.5 * u * u) for i in range(9)])
    gen = torch.Generator(device=device).manual_seed(seed)
    r = torch.rand((9, p["ny"], p["nx"]), generator=gen, dtype=torch.float64, device=device)
    return feq[:, :, None] * (1.0 + 1e-3 * (2.0 * r - 1.0))


# ---------------------------------------------------------------- the cases


def _host(shape):
    return torch.empty(shape, dtype=torch.float64, pin_memory=True).numpy()


def _batch_populations(b, d, out):
    """One domain's state through the C ABI into the caller's pinned memory
    (the binding's method allocates a new array on each call)."""
    binding._bcheck(binding.lib().lbm_batch_populations(b._h, d, binding._dp(out)), b._h)
    return out


def prepare(case, seed):
    kind = case["kind"]
    if kind == "sweep":
        ps = _sweep(case, seed)
        b = binding.Batch([dict(mask=_mask(p), tau=p["tau"], u_in=p["u"]) for p in ps], storage=case["storage"])
        b.autotune(trials=3)
        b.prepare(case["steps"])
        return dict(case=case, batch=b, outs=[_host((9, p["ny"], p["nx"])) for p in ps])
    if kind == "porous":
        mask, u, force = _discs(case, seed)
        lat = binding.Lattice(mask, case["tau"], u, kind=binding.PERIODIC, storage=case["storage"], body_force=force,
                              cv=[0, case["nx"] - 1, 0, case["ny"] - 1])
        lat.prepare(case["steps"])
        return dict(case=case, lat=lat, out=_host((9, case["ny"], case["nx"])))
    p = _section(case, seed)
    if kind == "job":
        return dict(case=case, p=p, out=_host((9, case["ny"], case["nx"])))
    lat = binding.Lattice(_mask(p), p["tau"], p["u"], storage=case["storage"])
    if kind == "grad":
        lat.set_populations(_start(p, seed, "cuda").cpu().numpy())
        return dict(case=case, lat=lat)
    lat.prepare(case["steps"])
    return dict(case=case, lat=lat, out=_host((9, case["ny"], case["nx"])))


def run(state):
    case = state["case"]
    kind, n = case["kind"], case["steps"]
    if kind == "monitor":
        lat = state["lat"]
        f = np.empty((2, n))
        for k in range(n):
            lat.step(1)
            f[:, k] = lat.force("B")
        return {"B": f, "populations": lat.populations(state["out"])}
    if kind == "sweep":
        b = state["batch"]
        t = b.steps_done
        b.step(n)
        every = range(b.num_domains)
        return {"forces": [np.stack([np.stack(b.force_series(d, s, t, n)) for s in BATCH_SCHEMES]) for d in every],
                "populations": [_batch_populations(b, d, state["outs"][d]) for d in every]}
    if kind == "grad":
        J, dtau, du, df0 = state["lat"].adjoint(n, case["window"], 1.0, 0.25, df0_device=True)
        # gradients of FP32 parameters, as an optimiser takes them
        return {"J": J, "dtau": np.float32(dtau), "du": du.astype(np.float32), "df0": df0.to(torch.float32)}
    if kind == "job":
        p = state["p"]
        lat = binding.Lattice(_mask(p), p["tau"], p["u"], storage=case["storage"])
        lat.step(n)
        forces = np.stack([np.stack(lat.force_series(s)) for s in SCHEMES])
        cd, cl, stats = lat.coefficients("B", p["chord"], U0, n // 2, n - n // 2)
        pop = lat.populations(state["out"])
        lat.close()
        return {"forces": forces, "cd": cd, "cl": cl, "stats": np.array(stats), "populations": pop}
    lat = state["lat"]
    t = lat.steps_done
    lat.step(n)
    return {"forces": np.stack([np.stack(lat.force_series(s, t, n)) for s in SCHEMES]),
            "populations": lat.populations(state["out"])}


def _nodes(case):
    if case["kind"] != "sweep":
        return case["nx"] * case["ny"]
    return sum(p["nx"] * p["ny"] for p in _sweep(case, 1))


def work(case):
    """The state read once and its results (the FP64 populations, or the FP64
    gradient of the start state) written once, and the collisions of every step.
    A gradient's steps count three times: the step, and its transpose's two
    products with the state and with the adjoint."""
    n, e = _nodes(case), ELEM[case["storage"]]
    passes = 3 if case["kind"] == "grad" else 1
    return {"bytes": float(n * 9 * (e + 8)), "flops": float(passes * FLOPS_PER_UPDATE * n * case["steps"])}


# ---------------------------------------------------------------- the same in torch FP64

CX = (0, 1, 0, -1, 0, 1, -1, -1, 1)
CY = (0, 0, 1, 0, -1, 1, 1, -1, -1)
OPP = (0, 3, 4, 1, 2, 7, 8, 5, 6)
W = (4 / 9,) + (1 / 9,) * 4 + (1 / 36,) * 4


def _plain_mask(p):
    """The body from its closed form, rounded in the order that include/gblbm.h states."""
    x = np.arange(p["nx"], dtype=np.float64)[None, :]
    y = np.arange(p["ny"], dtype=np.float64)[:, None]
    dx, dy, c = x - p["xc"], y - p["yc"], p["chord"]
    if p["body"] == "cylinder":
        return (dx * dx + dy * dy <= (0.5 * c) * (0.5 * c)).astype(np.uint8)
    a = p["alpha"] * math.pi / 180.0
    ca, sa = math.cos(a), math.sin(a)
    xi, eta = (dx * ca - dy * sa) + 0.5 * c, dx * sa + dy * ca
    s = np.clip(xi, 0.0, c) / c
    yt = 0.2969 * np.sqrt(s) - 0.1260 * s
    yt = yt - 0.3516 * s * s
    yt = yt + 0.2843 * s * s * s
    yt = yt - 0.1015 * s * s * s * s
    yt = 5.0 * p["thickness"] * c * yt
    return ((xi >= 0.0) & (xi <= c) & (np.abs(eta) <= yt)).astype(np.uint8)


class _Plain:
    """One domain in FP64: collide, stream with halfway bounce-back, inlet and outlet."""

    def __init__(self, mask, tau, u, periodic=False, force=(0.0, 0.0)):
        self.solid = torch.from_numpy(mask.astype(bool)).cuda()
        self.ny, self.nx = mask.shape
        self.om, self.periodic, self.force = 1.0 / tau, periodic, force
        self.u = torch.from_numpy(np.ascontiguousarray(u, np.float64)).cuda()
        self.w = torch.tensor(W, dtype=torch.float64, device="cuda")
        self.bounce = [torch.roll(self.solid, (CY[i], CX[i]), (0, 1)) & ~self.solid for i in range(9)]
        node, way = [], []
        for i in range(1, 9):
            at = torch.nonzero((self.bounce[OPP[i]]).reshape(-1)).reshape(-1)
            node.append(at)
            way.append(torch.full_like(at, i))
        self.node, self.way = torch.cat(node), torch.cat(way)
        cx, cy = (torch.tensor(v, dtype=torch.float64, device="cuda") for v in (CX, CY))
        self.c = torch.stack([cx[self.way], cy[self.way]])
        N = self.nx * self.ny
        self.out_at = self.way * N + self.node
        self.back_at = torch.tensor(OPP, device="cuda")[self.way] * N + self.node
        self.axis = self.node[self.way <= 4]
        self.axis_c = self.c[:, self.way <= 4]
        self.cc = [torch.tensor([a[i] * b[i] for i in range(9)], dtype=torch.float64, device="cuda")
                   for a, b in ((CX, CX), (CY, CY), (CX, CY))]
        self.cx, self.cy = cx, cy

    def inlet(self, u):
        return torch.stack([W[i] * (1.0 + 3.0 * CX[i] * u + 4.5 * (CX[i] * u) ** 2 - 1.5 * u * u) for i in range(9)])

    def start(self):
        f = self.inlet(self.u)[:, :, None].expand(9, self.ny, self.nx).clone()
        return self.fill(f)

    def fill(self, f):
        return torch.where(self.solid, self.w[:, None, None], f)

    def collide(self, f, om, u):
        rho = f.sum(0)
        jx = f[1] - f[3] + f[5] - f[6] - f[7] + f[8]
        jy = f[2] - f[4] + f[5] + f[6] - f[7] - f[8]
        ux, uy = jx / rho, jy / rho
        base = 1.0 - 1.5 * (ux * ux + uy * uy)
        post = []
        for i in range(9):
            cu = CX[i] * ux + CY[i] * uy if CX[i] and CY[i] else (CX[i] * ux if CX[i] else (CY[i] * uy if CY[i] else 0.0 * ux))
            v = f[i] + om * (W[i] * rho * (base + cu * (3.0 + 4.5 * cu)) - f[i])
            g = 3.0 * W[i] * (CX[i] * self.force[0] + CY[i] * self.force[1])
            post.append(v + g if g else v)
        post = torch.stack(post)
        if not self.periodic:
            post = torch.cat([self.inlet(u)[:, :, None], post[:, :, 1:]], 2)
        return post

    def stream(self, post, u):
        f = torch.stack([post[i] if i == 0 else
                         torch.where(self.bounce[i], post[OPP[i]], torch.roll(post[i], (CY[i], CX[i]), (0, 1)))
                         for i in range(9)])
        if not self.periodic:
            f = torch.cat([self.inlet(u)[:, :, None], f[:, :, 1:-1], f[:, :, -2:-1]], 2)
        return self.fill(f)

    def forces(self, f, post):
        """A, B, DRTT, A' and SI of one step: [5][2].  DRTT over a box that holds
        the whole body equals B (bounce-back, Section II), less the momentum that
        the body force adds to the box's fluid."""
        f1, p1 = f.reshape(-1), post.reshape(-1)
        fi, fo, pi = f1[self.out_at], f1[self.back_at], p1[self.out_at]
        A, B, R = self.c @ (fi + fo), self.c @ (2.0 * pi), self.c @ (fi + pi)
        fluid = float((~self.solid).sum()) if self.periodic else 0.0
        D = B - fluid * torch.tensor(self.force, dtype=torch.float64, device="cuda")
        a = f.reshape(9, -1)[:, self.axis]
        rho, jx, jy = a.sum(0), self.cx @ a, self.cy @ a
        ux, uy = jx / rho, jy / rho
        visc = 1.0 - 0.5 * self.om
        sxx = visc * (self.cc[0] @ a - rho / 3.0 - rho * ux * ux)
        syy = visc * (self.cc[1] @ a - rho / 3.0 - rho * uy * uy)
        sxy = visc * (self.cc[2] @ a - rho * ux * uy)
        nx, ny, p = self.axis_c[0], self.axis_c[1], rho / 3.0
        S = torch.stack([(nx * (p + sxx) + ny * sxy).sum(), (nx * sxy + ny * (p + syy)).sum()])
        return torch.stack([A, B, D, R, S])

    def steps(self, f, n):
        F = []
        for _ in range(n):
            post = self.collide(f, self.om, self.u)
            F.append(self.forces(f, post))
            f = self.stream(post, self.u)
        return torch.where(self.solid, 0.0, f), torch.stack(F, 2)

    def gradient(self, f, n, window, wx, wy):
        kept = []
        J = 0.0
        wv = torch.tensor((wx, wy), dtype=torch.float64, device="cuda") / window
        for t in range(n):
            kept.append(f)
            post = self.collide(f, self.om, self.u)
            if t >= n - window:
                J += float(wv @ (self.c @ (2.0 * post.reshape(-1)[self.out_at])))
            f = self.stream(post, self.u)
        lam = torch.zeros_like(f)
        dom, du = 0.0, torch.zeros_like(self.u)
        for t in reversed(range(n)):
            f = kept.pop().requires_grad_(True)
            om = torch.tensor(self.om, dtype=torch.float64, device="cuda", requires_grad=True)
            u = self.u.clone().requires_grad_(True)
            post = self.collide(f, om, u)
            # the inlet velocity enters through the inlet's post-collision state
            L = (self.stream(post, u.detach()) * lam).sum()
            if t >= n - window:
                L = L + wv @ (self.c @ (2.0 * post.reshape(-1)[self.out_at]))
            lam, go, gu = torch.autograd.grad(L, (f, om, u))
            dom += float(go)
            du += gu
        lam = torch.where(self.solid, 0.0, lam)
        lam[:, :, 0] = 0.0
        return J, -dom * self.om * self.om, du, lam


def exact(case, seed):
    kind, n = case["kind"], case["steps"]
    with torch.no_grad():
        if kind == "sweep":
            sims = [_Plain(_plain_mask(p), p["tau"], p["u"]) for p in _sweep(case, seed)]
            done = [s.steps(s.start(), n) for s in sims]
            at = [SCHEMES.index(s) for s in BATCH_SCHEMES]
            return {"forces": [F[at] for _, F in done], "populations": [f for f, _ in done]}
        if kind == "porous":
            mask, u, force = _discs(case, seed)
            s = _Plain(mask, case["tau"], u, True, force)
        else:
            p = _section(case, seed)
            s = _Plain(_plain_mask(p), p["tau"], p["u"])
    if kind == "grad":
        J, dtau, du, df0 = s.gradient(s.fill(_start(p, seed, "cuda")), n, case["window"], 1.0, 0.25)
        return {"J": J, "dtau": dtau, "du": du, "df0": df0}
    with torch.no_grad():
        f, F = s.steps(s.start(), n)
    if kind == "monitor":
        return {"B": F[1], "populations": f}
    if kind == "job":
        k = 2.0 / (U0 * U0 * p["chord"])
        cd, cl = k * F[1, 0, n // 2:], k * F[1, 1, n // 2:]
        stats = torch.stack([cd.mean(), cl.mean(), cd.std(unbiased=False), cl.std(unbiased=False)])
        return {"forces": F, "cd": cd, "cl": cl, "stats": stats, "populations": f}
    return {"forces": F, "populations": f}
