"""The work that users of this framework have it do, as measurable cases.

A case is one model step of the ray-volume tracer (with its sources, its background and its output
buffers as the program around it has them), one inference of the drag surrogate or one stretch of
its training.  `listed()` names the cases, `draw()` makes more of the same ranges, `prepare()` makes
what a program holds before the call, `run()` is one pass through the public entry points, `work()`
counts what a pass cannot do without and `exact()` gives the same outputs in plain 64-bit torch.
"""
import math

import numpy as np
import torch

from paper_2309_11257_gb300 import gwam, synth

N_IN, N_OUT, NLEV = 368, 180, 90      # the surrogate's columns: four fields on 90 levels and 8 source values


def listed():
    step = dict(kind="step", members=1, columnar=0, theta=0, flux_form=0, physics=1, cap=4800, background="fixed", call="graph",
                dt=60.0, spinup=40)
    sphere = dict(step, grid="sphere", nx=256, ny=128, nz=90, precision=0, source="once")
    return [
        # the smallest call in use: a regional box (the f-plane configuration's size) that a convection
        # scheme feeds every step, about 4096 ray volumes; launches and latency are all of it
        dict(step, name="box_storms", grid="box", nx=16, ny=16, nz=64, precision=0, source="storms", physics=0, cap=16,
             call="step", dt=300.0),
        # a coarse global model with continuous ghost-layer emission under a small cap, odd sizes
        dict(step, name="sphere_ghost_small", grid="sphere", nx=45, ny=23, nz=31, precision=0, source="ghost", cap=40),
        # a mid-size global grid of ragged sizes in the precision form with the pseudomomentum fluxes
        dict(step, name="sphere_ragged_fp32", grid="sphere", nx=131, ny=67, nz=61, precision=1, source="once", flux_form=1),
        # the benchmark's sphere in the FP64 form, waves aloft
        dict(sphere, name="sphere_fp64"),
        # the benchmark's larger sphere in the precision form
        dict(sphere, name="sphere_fp32", nx=512, ny=256, precision=1),
        # a small ensemble of spheres, each with its own background, background and convective sources
        dict(sphere, name="ensemble_fp64", nx=128, ny=64, members=4, source="once+storms"),
        # operational use: the source emits through the ghost layer before every 60 s step, the cap holds
        # the population
        dict(sphere, name="sphere_ghost", nx=128, ny=64, source="ghost", cap=96),
        # online coupling: the host model advances u, v by the drag and sets the background every step;
        # the potential-temperature flux is projected too
        dict(sphere, name="sphere_coupled", background="coupled", theta=1, call="step"),
        # a CPU host model: background up and drag down the host link every step
        dict(sphere, name="sphere_host", background="host", call="host"),
        # the drag surrogate in place of the tracer: the columns of one 256 x 128 sphere
        dict(name="infer_sphere", kind="infer", ncol=32768, hidden=512, layers=4),
        # the same for a regional model's few columns
        dict(name="infer_few", kind="infer", ncol=1000, hidden=512, layers=4),
        # training the surrogate: a stretch of Adam steps of 4096 columns between two reads of the weights
        dict(name="train", kind="train", batch=4096, steps=16, rows=65536, hidden=512, layers=4),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step"] * 8 + ["infer", "infer", "train"])
    net = dict(hidden=rng.choice([128, 256, 512, 512, 512]), layers=rng.choice([2, 3, 4, 4, 4]))
    if kind == "infer":
        return dict(net, kind="infer", ncol=_log_int(rng, 1, 131072))
    if kind == "train":
        return dict(net, kind="train", batch=64 * _log_int(rng, 1, 64), steps=rng.randint(1, 16), rows=_log_int(rng, 2000, 131072))
    c = dict(kind="step", members=1, columnar=int(rng.random() < 0.15), theta=int(rng.random() < 0.2),
             flux_form=int(rng.random() < 0.2), physics=int(rng.random() < 0.9), cap=4800, background="fixed",
             call=rng.choice(["graph", "graph", "step"]), spinup=rng.randint(2, 40), precision=rng.choice([0, 0, 1]))
    if rng.random() < 0.2:
        n = _log_int(rng, 8, 80)
        c.update(grid="box", nx=n, ny=max(4, int(n * rng.uniform(0.5, 1.5))), nz=rng.randint(20, 80), dt=300.0,
                 source=rng.choice(["once", "storms"]))
        if c["source"] == "storms":
            c["cap"] = rng.randint(8, 48)
    else:
        n = _log_int(rng, 24, 300)
        c.update(grid="sphere", nx=n, ny=max(12, int(n * rng.uniform(0.4, 0.6))), nz=rng.randint(24, 100), dt=60.0,
                 source=rng.choice(["once", "once", "ghost", "once+storms"]))
        if c["source"] == "ghost":
            c["cap"] = rng.randint(24, 120)
        c["background"] = rng.choice(["fixed"] * 4 + ["coupled", "host"])
        if c["background"] == "host":
            c["call"] = "host"
        elif n <= 100:
            c["members"] = rng.choice([1, 1, 2, 3])
    if c["members"] > 1:
        c["background"] = "fixed"
    return c


# ------------------------------------------------------------------ inputs (host, from the seed)

def _grid(c):
    if c["grid"] == "box":
        return synth.fplane_grid(nx=c["nx"], ny=c["ny"], nz=c["nz"])
    return synth.sphere_grid(nx=c["nx"], ny=c["ny"], nz=c["nz"], dz=1000.0)


def _params(c):
    return dict(synth.DEFAULT_PARAMS, saturation=c["physics"], smoothing=c["physics"], flux_form=c["flux_form"],
                cap_per_column=c["cap"], columnar=c["columnar"], theta_flux=c["theta"])


def _backgrounds(c, seed):
    """The members' U, V, N^2, rho on the GPU: the workloads' analytic states plus a smooth seeded perturbation."""
    g = synth.rng(20_000_000 + seed)
    grid, out = _grid(c), []
    x, y, z = (torch.from_numpy(a).cuda() for a in synth.node_coords(grid))
    for _ in range(c["members"]):
        one = torch.ones((c["nz"], c["ny"], c["nx"]), dtype=torch.float64, device="cuda")
        amp, lat, ph = g.uniform(50.0, 70.0), g.uniform(40.0, 50.0), g.uniform(0.0, 2.0 * math.pi, 8)
        xx = torch.arange(c["nx"], dtype=torch.float64, device="cuda")[None, None, :] * (2.0 * math.pi / c["nx"])
        yy = torch.linspace(0.0, 1.0, c["ny"], dtype=torch.float64, device="cuda")[None, :, None]
        zz = torch.linspace(0.0, 1.0, c["nz"], dtype=torch.float64, device="cuda")[:, None, None]
        if c["grid"] == "box":
            u0, n2c, h, rho0 = 10.0 * one, 4e-4, 7000.0, 1.2
        else:
            n2c, h, rho0 = synth.isothermal()
            deg = torch.rad2deg(y)
            lats = torch.exp(-((deg - lat) / 10.0) ** 2) + torch.exp(-((deg + lat) / 10.0) ** 2)
            u0 = amp * torch.exp(-((z - 60e3) / 15e3) ** 2)[:, None, None] * lats[None, :, None] * one
        u = u0 + 5.0 * torch.sin(xx + ph[0]) * torch.cos(3 * yy + ph[1]) * torch.sin(2 * zz + ph[2])
        v = 3.0 * one * torch.cos(2 * xx + ph[3]) * torch.sin(2 * yy + ph[4]) * torch.cos(zz + ph[5])
        n2 = n2c * (1.0 + 0.05 * torch.sin(xx + ph[6]) * torch.cos(4 * yy + ph[2]) * torch.cos(3 * zz + ph[3]))
        rho = rho0 * torch.exp(-z / h)[:, None, None] * (1.0 + 0.05 * torch.cos(xx + ph[7]) * torch.sin(2 * yy + ph[5]) * one)
        out.append([f.contiguous() for f in (u, v, n2, rho)])
    return out


def _specs(c, seed):
    """Convective launches: in every tenth column or so (once+storms: a lognormal number in every column)."""
    grid, out = _grid(c), []
    for m in range(c["members"]):
        once = c["source"] == "once+storms"
        sp = synth.convective_specs(grid, tag=30_000_000 + 300 * seed + m, median=16.0 if once else 3.0, sigma=1.0,
                                    cap=512 if once else 12, col_fraction=1.0 if once else 0.25, z_launch=10e3 if once else 5e3)
        sp["member"] = m
        out.append(sp)
    return np.concatenate(out)


def _rays(c, seed):
    """Explicit ray volumes of a box: 16 a column, as the f-plane configuration has them."""
    return synth.fplane_rays(_grid(c), 16 * c["nx"] * c["ny"], tag=40_000_000 + seed)


def _columns(c):
    """Columns that the background source launches into (|phi| <= 85 degrees)."""
    _, phi, _ = synth.node_coords(_grid(c))
    return c["nx"] * int((np.abs(np.degrees(phi)) <= 85.0).sum())


def _rays_about(c):
    if c["source"] == "ghost":
        return _columns(c) * min(c["cap"], 32 * (c["spinup"] + 1))
    if c["grid"] == "box":
        return 16 * c["nx"] * c["ny"]
    return c["members"] * _columns(c) * (32 + (26 if c["source"] == "once+storms" else 0))


def _network(c, seed):
    g = np.random.Generator(np.random.PCG64(50_000_000 + seed))
    dims = (N_IN,) + (c["hidden"],) * c["layers"] + (N_OUT,)
    par = [((g.standard_normal((o, i)) / math.sqrt(i)).astype(np.float32), (0.1 * g.standard_normal(o)).astype(np.float32))
           for i, o in zip(dims[:-1], dims[1:])]
    norm = [g.uniform(-1, 1, N_IN), g.uniform(0.5, 2, N_IN), 1e-5 * g.uniform(-1, 1, N_OUT), np.full(N_OUT, 3e-5),
            np.full(N_IN, -4.2), np.full(N_IN, 4.2)]
    return par, [a.astype(np.float32) for a in norm]


def _data(c, seed, n):
    """n columns of features and targets on the GPU, normal about the normalisation's mean."""
    _, (xm, xs, ym, ys, _, _) = _network(c, seed)
    g = torch.Generator(device="cuda").manual_seed(60_000_000 + seed)
    mu, sg, tm, ts = (torch.from_numpy(a).cuda() for a in (xm, xs, ym, ys))
    X = torch.randn((n, N_IN), generator=g, device="cuda") * sg + mu
    Y = torch.randn((n, N_OUT), generator=g, device="cuda") * ts + tm
    return X, Y


# ------------------------------------------------------------------ prepare and run

def prepare(case, seed):
    c = case
    if c["kind"] != "step":
        par, norm = _network(c, seed)
        n = c["ncol"] if c["kind"] == "infer" else c["rows"]
        X, Y = _data(c, seed, n)
        S = gwam.Surrogate(n_hidden=c["hidden"], n_layers=c["layers"], max_batch=32768 if c["kind"] == "infer" else 8192)
        S.set_normalization(*norm)
        S.set_params(par)
        st = dict(case=c, S=S, X=X, Y=Y, seed=seed)
        if c["kind"] == "infer":
            st.update(du=torch.zeros((NLEV, n), dtype=torch.float64, device="cuda"),
                      dv=torch.zeros((NLEV, n), dtype=torch.float64, device="cuda"),
                      mask=torch.zeros(n, dtype=torch.int32, device="cuda"), nfb=torch.zeros(1, dtype=torch.int32, device="cuda"))
        return st
    grid, bg = _grid(c), _backgrounds(c, seed)
    T = gwam.Tracer(grid, dict(_params(c), precision=c["precision"]), max_rays=2 * _rays_about(c) + 64 * c["nx"] * c["ny"] + 4096,
                    members=c["members"])
    if c["members"] == 1:
        T.set_background(*bg[0])
    else:
        for m, b in enumerate(bg):
            T.set_member_background(m, *b)
    shape = (c["nz"], c["ny"], c["nx"]) if c["members"] == 1 else (c["members"], c["nz"], c["ny"], c["nx"])
    st = dict(case=c, T=T, bg=bg, src=synth.background_source())
    if c["call"] == "host":
        st["host_bg"] = [b.cpu().pin_memory() for b in bg[0]]
        st["host_out"] = [torch.zeros(shape, dtype=torch.float64).pin_memory() for _ in range(2)]
    st["du"] = torch.zeros(shape, dtype=torch.float64, device="cuda")
    st["dv"] = torch.zeros_like(st["du"])
    if "storms" in c["source"]:
        st["specs"] = _specs(c, seed)
    if c["source"].startswith("once"):
        T.add_rays(_rays(c, seed)) if c["grid"] == "box" else T.launch_sources(st["src"])
        if c["source"] == "once+storms":
            T.launch_spectral(st["specs"])
    # the lead-in: ray volumes spread over the levels, waves aloft
    for _ in range(c["spinup"]):
        _emit(st)
        T.step_graph(_lead_dt(c), st["du"], st["dv"])
    T.synchronize()
    return st


def _lead_dt(c):
    return c["dt"] if c["source"] in ("ghost", "storms") else 300.0


def _emit(st):
    c = st["case"]
    if c["source"] == "ghost":
        st["T"].launch_ghost(st["src"], c["dt"])
    elif c["source"] == "storms":
        st["T"].launch_spectral(st["specs"])


def run(st):
    c = st["case"]
    if c["kind"] == "infer":
        st["S"].infer(st["X"], st["du"], st["dv"], st["mask"], st["nfb"])
        return dict(du=st["du"], dv=st["dv"], mask=st["mask"], fallback=st["nfb"])
    if c["kind"] == "train":
        for it in range(c["steps"]):
            st["S"].train_step(st["X"], st["Y"], c["batch"], seed=st["seed"] * 1_000_003 + it, lr=1e-3)
        return dict(params=st["S"].params())
    T, du, dv = st["T"], st["du"], st["dv"]
    _emit(st)
    if c["background"] == "host":
        T.set_background_async(*[b.numpy() for b in st["host_bg"]])
        T.step_host_async(c["dt"], *[o.numpy() for o in st["host_out"]])
        return dict(dudt=st["host_out"][0], dvdt=st["host_out"][1])
    if c["background"] == "coupled":
        T.set_background(*st["bg"][0])
    (T.step_graph if c["call"] == "graph" else T.step)(c["dt"], du, dv)
    if c["background"] == "coupled":
        u, v = st["bg"][0][:2]
        u.add_(du, alpha=c["dt"])
        v.add_(dv, alpha=c["dt"])
        return dict(dudt=du, dvdt=dv, u=u, v=v)
    return dict(dudt=du, dvdt=dv)


def work(case):
    """A step: the background read once (4 FP64 fields), du/dt and dv/dt written, each ray volume's
    record read and written (13 FP64 values and an id; 64 bytes in the precision form), about 1460
    operations a ray volume.  A network: features in, drag out, weights once; 2 operations a weight
    and column, three times that in training."""
    c = case
    if c["kind"] == "step":
        rays, cells = _rays_about(c), c["members"] * c["nx"] * c["ny"] * c["nz"]
        return dict(bytes=rays * (128.0 if c["precision"] else 224.0) + cells * 48.0, flops=rays * 1460.0)
    dims = (N_IN,) + (c["hidden"],) * c["layers"] + (N_OUT,)
    weights = sum(a * b for a, b in zip(dims[:-1], dims[1:]))
    if c["kind"] == "infer":
        return dict(bytes=c["ncol"] * (4.0 * N_IN + 8.0 * N_OUT + 4.0) + 2.0 * weights, flops=2.0 * weights * c["ncol"])
    return dict(bytes=c["steps"] * (c["batch"] * 4.0 * (N_IN + N_OUT) + weights * 24.0), flops=6.0 * weights * c["batch"] * c["steps"])


# ------------------------------------------------------------------ the same in plain 64-bit torch

def exact(case, seed):
    c = case
    if c["kind"] == "infer":
        par, (xm, xs, ym, ys, lo, hi) = _network(c, seed)
        X, _ = _data(c, seed, c["ncol"])
        d = lambda a: torch.from_numpy(a).cuda().double()  # noqa: E731
        a = (X.double() - d(xm)) / d(xs)
        inside = ((a >= d(lo)) & (a <= d(hi))).all(1)
        y = _mlp([(d(W), d(b)) for W, b in par], a) * d(ys) + d(ym)
        y = torch.where(inside[:, None], y, torch.zeros_like(y)).t().contiguous()
        return dict(du=y[:NLEV].contiguous(), dv=y[NLEV:].contiguous(), mask=None, fallback=None)
    if c["kind"] == "train":
        return dict(params=_train64(c, seed))
    return _Model64(c, seed).outputs()


def _mlp(par, a):
    for q, (W, b) in enumerate(par):
        a = a @ W.t() + b
        if q < len(par) - 1:
            a = 0.5 * a * (1.0 + torch.erf(a / math.sqrt(2.0)))
    return a


def _train64(c, seed):
    par, (xm, xs, ym, ys, _, _) = _network(c, seed)
    X, Y = _data(c, seed, c["rows"])
    d = lambda a: torch.from_numpy(a).cuda().double()  # noqa: E731
    flat = [d(a).requires_grad_() for W, b in par for a in (W, b)]
    mom = [(torch.zeros_like(p), torch.zeros_like(p)) for p in flat]
    for t in range(1, c["steps"] + 1):
        s = np.uint64((seed * 1_000_003 + t - 1) % 2 ** 64)
        with np.errstate(over="ignore"):
            z = s + np.arange(1, c["batch"] + 1, dtype=np.uint64) * np.uint64(0x9E3779B97F4A7C15)
            z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
            z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
            rows = torch.from_numpy(((z ^ (z >> np.uint64(31))) % np.uint64(c["rows"])).astype(np.int64)).cuda()
        a, tgt = (X[rows].double() - d(xm)) / d(xs), (Y[rows].double() - d(ym)) / d(ys)
        loss = ((_mlp(list(zip(flat[::2], flat[1::2])), a) - tgt) ** 2).mean()
        for p, (m, v), g in zip(flat, mom, torch.autograd.grad(loss, flat)):
            m.mul_(0.9).add_(0.1 * g)
            v.mul_(0.999).add_(0.001 * g * g)
            with torch.no_grad():
                p.sub_(1e-3 * (m / (1 - 0.9 ** t)) / ((v / (1 - 0.999 ** t)).sqrt() + 1e-8))
    flat = [p.detach() for p in flat]
    return list(zip(flat[::2], flat[1::2]))


class _Model64:
    """The tracer's step in 64-bit torch, all ray volumes at once.  Fields are [members][nz][ny][nx] flat;
    the ray state s is a list of 13 vectors (x y z k l m ex ey ez px py pz n) beside id and member."""

    def __init__(self, c, seed):
        self.c, self.g, self.src = c, _grid(c), synth.background_source()
        self.sph = c["grid"] == "sphere"
        self.dX, self.dY = (2 * math.pi / c["nx"], math.pi / c["ny"]) if self.sph else (self.g["dx"], self.g["dy"])
        self.y0, self.dz = (-0.5 * math.pi if self.sph else 0.0), self.g["dz"]
        self.Lx, self.Ly, self.ztop = self.dX * c["nx"], self.dY * c["ny"], c["nz"] * self.dz
        self.bg = _backgrounds(c, seed)
        self.set_background()
        self.s = [torch.zeros(0, dtype=torch.float64, device="cuda") for _ in range(13)]
        self.id = torch.zeros(0, dtype=torch.int64, device="cuda")
        self.mem = torch.zeros(0, dtype=torch.int64, device="cuda")
        self.next_id = 0
        specs = _specs(c, seed) if "storms" in c["source"] else None
        if c["source"].startswith("once"):
            self.add(_rays(c, seed)) if c["grid"] == "box" else self.launch(self.bins(), 0.0)
            if specs is not None:
                self.launch(self.spec_bins(specs), 0.0)
        for q in range(c["spinup"] + 1):
            if c["source"] == "ghost":
                self.launch(self.bins(), c["dt"])
            elif c["source"] == "storms":
                self.launch(self.spec_bins(specs), 0.0)
            self.step(c["dt"] if q == c["spinup"] else _lead_dt(c))

    def outputs(self):
        c = self.c
        out = dict(dudt=self.du[0] if c["members"] == 1 else self.du, dvdt=self.dv[0] if c["members"] == 1 else self.dv)
        if c["background"] == "coupled":
            out.update(u=self.bg[0][0] + c["dt"] * self.du[0], v=self.bg[0][1] + c["dt"] * self.dv[0])
        return out

    # -- background: node values and centred differences, interpolated trilinearly, held outside the edge nodes
    def set_background(self):
        F = [torch.stack([b[q] for b in self.bg]) for q in range(4)]
        U, V, N2, self.rho = F
        lr = torch.log(self.rho)
        G2 = 0.25 * self.along(lr, 1, False, self.dz) ** 2
        self.nodes = torch.stack([torch.stack([a, self.along(a, 3, True, self.dX), self.along(a, 2, not self.sph, self.dY),
                                               self.along(a, 1, False, self.dz)]) for a in (U, V, N2, G2)]).reshape(16, -1)

    @staticmethod
    def along(a, dim, periodic, h):
        if periodic:
            return (torch.roll(a, -1, dim) - torch.roll(a, 1, dim)) / (2 * h)
        n, s = a.shape[dim], lambda lo, ln: a.narrow(dim, lo, ln)
        return torch.cat([(s(1, 1) - s(0, 1)) / h, (s(2, n - 2) - s(0, n - 2)) / (2 * h), (s(n - 1, 1) - s(n - 2, 1)) / h], dim)

    @staticmethod
    def bracket(u, n, periodic):
        if periodic:
            u = u - n * torch.floor(u / n)
            f = torch.floor(u)
            a = f.long() % n
            return a, (a + 1) % n, u - f
        f = torch.floor(u).clamp(0, n - 2)
        return f.long(), f.long() + 1, (u - f).clamp(0.0, 1.0)

    def gather(self, x, y, z, mem, which):
        c = self.c
        i, j, k = (self.bracket(x / self.dX - 0.5, c["nx"], True), self.bracket((y - self.y0) / self.dY - 0.5, c["ny"], not self.sph),
                   self.bracket(z / self.dz - 0.5, c["nz"], False))
        out = [torch.zeros_like(x) for _ in which]
        for a in range(2):
            for b in range(2):
                for e in range(2):
                    w = (i[2] if a else 1 - i[2]) * (j[2] if b else 1 - j[2]) * (k[2] if e else 1 - k[2])
                    at = ((mem * c["nz"] + k[e]) * c["ny"] + j[b]) * c["nx"] + i[a]
                    for o, f in zip(out, which):
                        o += w * self.nodes[f][at]
        return out

    # -- ray equations
    def coriolis(self, y):
        if not self.sph:
            return torch.full_like(y, self.g["f0"]), torch.zeros_like(y)
        w = self.g["omega"]
        return 2 * w * torch.sin(y), 8 * w * w * torch.sin(y) * torch.cos(y)

    @staticmethod
    def disp(kh2, mg2, n2, f2):
        K2, D = kh2 + mg2, n2 - f2
        w2 = (f2 * mg2 + n2 * kh2) / K2
        w = torch.sqrt(w2)
        return K2, D, w, D / (w * K2 * K2)

    def rates(self, s, mem, columnar):
        x, y, z, k, l, m = s[:6]
        b = self.gather(x, y, z, mem, range(16))
        val, grad = b[0::4], [b[4 * f + 1:4 * f + 4] for f in range(4)]
        f, df2 = self.coriolis(y)
        f2, zero = f * f, torch.zeros_like(x)
        df = [zero, df2, zero]
        r = self.g["radius"] + z if self.sph else torch.ones_like(x)
        hX = r * torch.cos(y) if self.sph else r
        kh2, m2 = k * k + l * l, m * m
        mg2 = m2 + val[3]
        K2, D, w, cc = self.disp(kh2, mg2, val[2], f2)
        cg = [k * mg2 * cc + val[0], l * mg2 * cc + val[1], -m * kh2 * cc]
        G = [k * grad[0][q] + l * grad[1][q] + kh2 / (2 * w * K2) * (grad[2][q] - D / K2 * grad[3][q]) + mg2 / (2 * w * K2) * df[q]
             for q in range(3)]
        if columnar:
            R = [zero, zero, zero, zero, zero, -G[2]]
        elif self.sph:
            t = torch.tan(y)
            R = [zero] * 3 + [-G[0] / hX - k * cg[2] / r + k * t * cg[1] / r, -G[1] / r - l * cg[2] / r - k * t * cg[0] / r,
                              -G[2] + k * cg[0] / r + l * cg[1] / r]
        else:
            R = [zero] * 3 + [-a for a in G]
        R += [zero] * 3
        for q in range(3):
            if columnar and q < 2:
                continue
            vel = []
            for h in (0.5 * s[6 + q], -0.5 * s[6 + q]):
                mgf = m2 + val[3] + grad[3][q] * h
                cf = self.disp(kh2, mgf, val[2] + grad[2][q] * h, f2 + df[q] * h)[3]
                if q == 0:
                    vel.append((k * mgf * cf + val[0] + grad[0][0] * h) / hX)
                elif q == 1:
                    vel.append((l * mgf * cf + val[1] + grad[1][1] * h) / r)
                else:
                    vel.append(-m * kh2 * cf)
            R[q], R[6 + q] = 0.5 * (vel[0] + vel[1]), vel[0] - vel[1]
        return R

    def rk3(self, s, mem, dt, columnar):
        s, p = list(s), [0.0] * 9
        for A, B in ((0.0, 1 / 3), (-5 / 9, 15 / 16), (-153 / 128, 8 / 15)):
            R = self.rates(s, mem, columnar)
            p = [A * a + dt * f for a, f in zip(p, R)]
            s = [a + B * b for a, b in zip(s[:9], p)] + s[9:]
        return s

    # -- sources
    def alpha(self, p):
        up = 0.5 * (1 - torch.cos(math.pi * (p - 20) / 30))
        return torch.where(p >= 80, (1 - (p - 80) / 5).clamp(0, 1), torch.where(p >= 50, torch.ones_like(p), torch.where(p >= 20, up, 0 * p)))

    def bins(self):
        c, s = self.c, self.src
        nb = s["n_az"] * s["n_c"]
        t = torch.arange(c["members"] * c["ny"] * c["nx"] * nb, device="cuda")
        col, q = t // nb, t % nb
        mem, col = col // (c["ny"] * c["nx"]), col % (c["ny"] * c["nx"])
        j, i = col // c["nx"], col % c["nx"]
        deg = (self.y0 + (j.double() + 0.5) * self.dY) * (180 / math.pi)
        tau = s["tau"]
        sp, sm = (self.alpha(p) * s["f_s"] + self.alpha(-p) * s["f_w"] for p in (deg, -deg))
        flux = 0.5 * (sp * (1 + math.cos(tau)) + sm * (1 - math.cos(tau))) / nb
        ok = deg.abs() <= s["phi_max_deg"]
        one = torch.ones_like(deg)
        b = dict(i=i, j=j, mem=mem, z=s["z_launch"] * one, d=s["dz_launch"] * one, th=2 * math.pi * (q // s["n_c"]).double() / s["n_az"],
                 cp=s["c_min"] * (s["c_max"] / s["c_min"]) ** ((q % s["n_c"]).double() / (s["n_c"] - 1)), lam=s["lambda_h"] * one,
                 flux=flux, frac=s["spectral_frac"] * one)
        return {n: a[ok] for n, a in b.items()}

    def spec_bins(self, sp):
        names = dict(i="i", j="j", mem="member", z="z_launch", d="dz_launch", th="theta", cp="c", lam="lambda_h", flux="flux", frac="spectral_frac")
        b = {n: torch.from_numpy(np.ascontiguousarray(sp[f])).cuda() for n, f in names.items()}
        return {n: a.long() if n in ("i", "j", "mem") else a for n, a in b.items()}

    def launch(self, b, ghost_dt):
        x, y, z = (b["i"].double() + 0.5) * self.dX, self.y0 + (b["j"].double() + 0.5) * self.dY, b["z"] + 0.5 * b["d"]
        U, V, N2, G2 = self.gather(x, y, z, b["mem"], (0, 4, 8, 12))
        f2 = self.coriolis(y)[0] ** 2
        kh = 2 * math.pi / b["lam"]
        k, l = kh * torch.cos(b["th"]), kh * torch.sin(b["th"])
        w = kh * b["cp"] - (k * U + l * V)
        m2 = kh * kh * (N2 - w * w) / (w * w - f2) - G2
        ok = (w > 0) & (w * w > f2) & (w * w < N2) & (m2 > 0)
        m = -torch.sqrt(m2.abs())
        cr = -m * kh * kh * self.disp(kh * kh, m2 + G2, N2, f2)[3]
        r = self.g["radius"] + z if self.sph else torch.ones_like(z)
        hX = r * torch.cos(y) if self.sph else r
        dk, dm, one = b["frac"] * kh, b["frac"] * m.abs(), torch.ones_like(x)
        s = [x, y, z, k, l, m, self.dX * one, self.dY * one, b["d"], hX * self.dX * dk, r * self.dY * dk, b["d"] * dm,
             b["flux"] / (kh * cr) / (dk * dk * dm)]
        s, mem, z0 = [a[ok] for a in s], b["mem"][ok], (b["z"] + b["d"])[ok]
        if ghost_dt > 0:
            e = self.rk3(s, mem, ghost_dt, True)
            top, bot = e[2] + 0.5 * e[8], e[2] - 0.5 * e[8]
            low = torch.maximum(bot, z0)
            s[11] = s[11] * (top - low) / e[8]
            s[2], s[5], s[8] = 0.5 * (low + top), e[5], top - low
            ok = (e[5] < 0) & (top > z0)
            s, mem = [a[ok] for a in s], mem[ok]
        ok = self.status(s) == 0
        self.append([a[ok] for a in s], mem[ok])

    def add(self, r):
        v = {n: torch.from_numpy(a).cuda() for n, a in r.items()}
        self.append([v["x"] % self.Lx, v["y"] % self.Ly, v["z"], v["k"], v["l"], v["m"], v["ex"], v["ey"], v["ez"], v["ex"] * v["dk"],
                     v["ey"] * v["dl"], v["ez"] * v["dm"], v["n"]], torch.zeros(len(r["x"]), dtype=torch.int64, device="cuda"))

    def append(self, s, mem):
        n = len(mem)
        self.s = [torch.cat([a, b]) for a, b in zip(self.s, s)]
        self.id = torch.cat([self.id, self.next_id + torch.arange(n, device="cuda")])
        self.mem = torch.cat([self.mem, mem])
        self.next_id += n

    # -- one step
    def status(self, s):
        bad = torch.zeros(len(s[0]), dtype=torch.bool, device="cuda")
        for a in s:
            bad |= ~torch.isfinite(a)
        bad |= ~((s[6] > 0) & (s[7] > 0) & (s[8] > 0))
        out = ~((s[2] >= 0) & (s[2] < self.ztop))
        if self.sph:
            out |= ~(s[1].abs() <= 0.5 * math.pi - 0.5 * self.dY)
        return torch.where(bad, 2, torch.where(out, 1, 0))

    def wrap(self, s):
        s[0] = s[0] - self.Lx * torch.floor(s[0] / self.Lx)
        if not self.sph:
            s[1] = s[1] - self.Ly * torch.floor(s[1] / self.Ly)
        return s

    def ijk(self, s):
        c = self.c
        return (torch.floor(s[0] / self.dX).clamp(0, c["nx"] - 1).long(), torch.floor((s[1] - self.y0) / self.dY).clamp(0, c["ny"] - 1).long(),
                torch.floor(s[2] / self.dz).clamp(0, c["nz"] - 1).long())

    def cosrow(self, j):
        return torch.cos(self.y0 + (j.double() + 0.5) * self.dY) if self.sph else torch.ones_like(j, dtype=torch.float64)

    def split(self, s):
        """Children (state, order among the parent's children, parent): vertical halves first, then horizontal ones."""
        n = len(s[0])
        kid, par = torch.zeros(n, dtype=torch.int64, device="cuda"), torch.arange(n, device="cuda")
        vert = s[8] > max(2.5 * self.dz, 1000.0)
        cr = self.cosrow(self.ijk(s)[1]) * self.dX * self.dY
        lx = torch.cos(s[1]) * s[6] if self.sph else s[6]
        hor = (lx > 2.5 * torch.sqrt(cr)) | (s[7] > 2.5 * torch.sqrt(cr)) | (lx * s[7] > 2.5 * cr)
        axis, nv = torch.where(lx >= s[7], 0, 1), vert.long() + 1
        for which in (vert, None):
            pick = (which if which is not None else hor)[par]
            ax = torch.full_like(par, 2) if which is not None else axis[par]
            hi = [a[pick].clone() for a in s]
            lo = [a.clone() for a in s]
            for q in range(3):
                at = pick & (ax == q)
                up = ax[pick] == q
                for t, sel, sign in ((lo, at, -0.25), (hi, up, 0.25)):
                    t[q] = torch.where(sel, t[q] + sign * t[6 + q], t[q])
                    t[6 + q], t[9 + q] = (torch.where(sel, 0.5 * t[e + q], t[e + q]) for e in (6, 9))
            kid_hi = kid[pick] + (1 if which is not None else nv[par[pick]])
            s, kid, par = [torch.cat([a, b]) for a, b in zip(lo, hi)], torch.cat([kid, kid_hi]), torch.cat([par, par[pick]])
        return self.wrap(s), kid, par, (vert.long() + 1) * (hor.long() + 1)

    def intrinsic(self, s):
        n2, g2 = self.gather(s[0], s[1], s[2], self.mem, (8, 12))
        f = self.coriolis(s[1])[0]
        kh2 = s[3] ** 2 + s[4] ** 2
        mg2 = s[5] ** 2 + g2
        return (f, n2, kh2, mg2) + self.disp(kh2, mg2, n2, f * f)

    def step(self, dt):
        c = self.c
        s = self.wrap(self.rk3(self.s, self.mem, dt, c["columnar"]))
        ok = self.status(s) == 0
        s, ids, mem = [a[ok] for a in s], self.id[ok], self.mem[ok]
        s, kid, par, nch = self.split(s)
        before = torch.cumsum(nch - 1, 0) - (nch - 1)
        ids = torch.where(kid == 0, ids[par], self.next_id + before[par] + kid - 1)
        self.next_id += int((nch - 1).sum())
        mem = mem[par]
        ok = self.status(s) == 0
        s, ids, mem = [a[ok] for a in s], ids[ok], mem[ok]
        i, j, k = self.ijk(s)
        cell = ((mem * c["ny"] + j) * c["nx"] + i) * c["nz"] + k
        o = torch.argsort(ids)
        o = o[torch.argsort(cell[o], stable=True)]
        self.s, self.id, self.mem, cell = [a[o] for a in s], ids[o], mem[o], cell[o]
        cell = self.cap(cell)
        s = self.s
        if c["physics"]:
            cell = self.saturate(cell, dt)
        self.project(cell)

    def cap(self, cell):
        col = cell // self.c["nz"]
        if not len(col) or int(torch.bincount(col).max()) <= self.c["cap"]:
            return cell
        s = self.s
        E = self.intrinsic(s)[6] * s[12] * s[9] * s[10] * s[11]
        o = torch.argsort(self.id)                       # most energetic first, equal ones by the smaller id
        o = o[torch.argsort(E[o], descending=True, stable=True)]
        o = o[torch.argsort(col[o], stable=True)]
        first = torch.searchsorted(col[o], col[o])
        keep = torch.zeros(len(col), dtype=torch.bool, device="cuda")
        keep[o] = torch.arange(len(o), device="cuda") - first < self.c["cap"]
        self.s, self.id, self.mem = [a[keep] for a in s], self.id[keep], self.mem[keep]
        return cell[keep]

    def volume(self, j, k):
        if not self.sph:
            return torch.full_like(j, self.dX * self.dY * self.dz, dtype=torch.float64)
        return (self.g["radius"] + (k.double() + 0.5) * self.dz) ** 2 * self.cosrow(j) * self.dX * self.dY * self.dz

    def saturate(self, cell, dt):
        s = self.s
        i, j, k = self.ijk(s)
        _, _, kh2, _, K2, _, w, _ = self.intrinsic(s)
        pj = s[5] ** 2 * kh2 / (w * K2) * s[12] * s[9] * s[10] * s[11] / self.volume(j, k)
        u, at = torch.unique_consecutive(cell, return_inverse=True)
        P, Q = torch.zeros(len(u), dtype=torch.float64, device="cuda"), torch.zeros(len(u), dtype=torch.float64, device="cuda")
        P.index_add_(0, at, pj)
        Q.index_add_(0, at, pj * K2)
        rho = self.rho.reshape(-1)[((self.mem * self.c["nz"] + k) * self.c["ny"] + j) * self.c["nx"] + i]
        kap = torch.where(Q[at] > 0, ((P[at] - 0.5 * rho) / (2 * dt * Q[at])).clamp(min=0.0), torch.zeros_like(rho))
        s[12] = s[12] * (1 - 2 * kap * K2 * dt).clamp(min=0.0)
        return cell

    def project(self, cell):
        c, s = self.c, self.s
        M, nx, ny, nz = c["members"], c["nx"], c["ny"], c["nz"]
        i, j, k = self.ijk(s)
        f, n2, kh2, mg2, K2, D, w, cc = self.intrinsic(s)
        kk, ll, W = s[3], s[4], s[12] * s[9] * s[10] * s[11]
        aw, f2, w2 = W / self.volume(j, k), f * f, w * w
        chx, chy, chr_ = kk * mg2 * cc, ll * mg2 * cc, -s[5] * kh2 * cc
        if c["flux_form"] == 0:
            iden = K2 / (D * kh2)                        # 1 / (w^2 - f^2)
            t = [(w2 * chx * kk + f2 * chy * ll) * iden, (w2 * chx * ll - f2 * chy * kk) * iden, (w2 * chy * kk - f2 * chx * ll) * iden,
                 (w2 * chy * ll + f2 * chx * kk) * iden, -f2 * n2 * chr_ * iden * kk, -f2 * n2 * chr_ * iden * ll]
            zc = w2 * chr_ * iden
        else:
            t, zc = [chx * kk, chx * ll, chy * kk, chy * ll, 0 * kk, 0 * kk], chr_
        at = ((self.mem * nz + k) * ny + j) * nx + i
        F = [torch.zeros(M * nz * ny * nx, dtype=torch.float64, device="cuda").index_add_(0, at, aw * a).reshape(M, nz, ny, nx) for a in t]
        Z = [torch.zeros(M * (nz + 1) * ny * nx, dtype=torch.float64, device="cuda") for _ in range(2)]
        wh = W / ((self.g["radius"] + s[2]) ** 2 if self.sph else 1.0) / s[8] / (self.cosrow(j) * self.dX * self.dY)
        lo, hi = s[2] - 0.5 * s[8], s[2] + 0.5 * s[8]
        k0 = torch.floor(lo / self.dz - 0.5).long()
        span = int((torch.ceil(hi / self.dz + 0.5).long() - k0).max()) if len(k0) else -1
        for q in range(span + 1):
            kq = k0 + q
            zq = kq.double() * self.dz
            ov = (torch.minimum(hi, zq + 0.5 * self.dz) - torch.maximum(lo, zq - 0.5 * self.dz)) / self.dz
            on = (ov > 0) & (kq >= 1) & (kq < nz)
            at = ((self.mem * (nz + 1) + kq) * ny + j) * nx + i
            for a, b in zip(Z, (kk, ll)):
                a.index_add_(0, at[on], (wh * ov * zc * b)[on])
        Z = [a.reshape(M, nz + 1, ny, nx) for a in Z]
        if c["physics"]:
            F, Z = [self.smooth(a) for a in F], [self.smooth(a) for a in Z]
        self.divergence(F, Z)

    def smooth(self, a):
        a = (torch.roll(a, 1, 3) + 2 * a + torch.roll(a, -1, 3)) / 4
        if not self.sph:
            return (torch.roll(a, 1, 2) + 2 * a + torch.roll(a, -1, 2)) / 4
        s, n = torch.cat([a[:, :, :1], a[:, :, :-1]], 2), torch.cat([a[:, :, 1:], a[:, :, -1:]], 2)
        return (s + 2 * a + n) / 4

    def divergence(self, F, Z):
        c = self.c
        jj = torch.arange(c["ny"], device="cuda")
        cr = self.cosrow(jj)[None, None, :, None]
        r = (self.g["radius"] + (torch.arange(c["nz"], device="cuda").double() + 0.5) * self.dz)[None, :, None, None] if self.sph else 1.0
        out = []
        for xf, yf, zf, ef in ((F[0], F[2], Z[0], F[4]), (F[1], F[3], Z[1], F[5])):
            div = (zf[:, 1:] - zf[:, :-1]) / self.dz
            if not c["columnar"]:
                dx = (torch.roll(xf, -1, 3) - torch.roll(xf, 1, 3)) / (2 * self.dX)
                yc = yf * cr
                if self.sph:
                    edge = torch.zeros_like(yc[:, :, :1])
                    dy = (torch.cat([yc[:, :, 1:], edge], 2) - torch.cat([edge, yc[:, :, :-1]], 2)) / (2 * self.dY)
                else:
                    dy = (torch.roll(yc, -1, 2) - torch.roll(yc, 1, 2)) / (2 * self.dY)
                div = div + (dx + dy) / (r * cr)
            out.append(-div / self.rho + ef / (self.g["g"] * self.rho))
        self.du, self.dv = out
