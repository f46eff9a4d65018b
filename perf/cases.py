"""The work a user of this framework has it do, as cases that can be timed.

Every case is one call sequence of a user's program through the public entry
points (``paper_1412_5170_gb300.lbm``: Lattice, Batch, WarmStartNet):

  lattice  initialise one lattice, advance it, take the new state (or the
           moments) out: what every run of the solver does;
  stats    the observables of a lattice with the velocity snapshot of a
           convergence check, as a run to steady state takes them;
  preset   a large run's start: the built-in initial field, the first
           observables and the populations it was given;
  batch    many independent lattices advanced together, then observed and
           (for droplets and slabs of a sweep) reduced to radial profiles;
  train    passes of the warm-start network over its training set;
  predict  the network's profiles for a held-out sweep.

``exact`` restates the model (D2Q9, Carnahan-Starling EOS, the hybrid
psi / psi^2 force, BGK with Guo, exact-difference, Shan-Chen or Li forcing,
MRT with Guo) and the network in plain 64-bit torch.
"""
import math

import numpy as np
import torch

from paper_1412_5170_gb300 import lbm

TC = 0.18727 / 0.4963 / 4.0            # critical temperature of the EOS with a = 1, b = 4, R = 1
RATES = dict(s_e=0.8, s_eps=0.8, s_q=1.1)
E = [(0, 0), (1, 0), (0, 1), (-1, 0), (0, -1), (1, 1), (-1, 1), (-1, -1), (1, -1)]
W = [4 / 9] + [1 / 9] * 4 + [1 / 36] * 4
NET = [5, 128, 128, 128, 64]           # the warm-start network's layers
SAMPLES = 64                           # radial samples of a density profile


def _lattice(name, nx, ny, precision, collision, forcing, field, T, tau, A, K, steps, size, out="state", source="device", cell=0):
    c = dict(kind="lattice", nx=nx, ny=ny, precision=precision, collision=collision, forcing=forcing, field=field, T=T, tau=tau,
             A=A, K=K, steps=steps, size=size, out=out, source=source, cell=cell)
    return dict(c, name=name) if name else c


def listed():
    return [
        # the plain method's case: a slab on 64 x 64 in FP64, its interfaces waved by half a node, host arrays in, moments out (the
        # smallest lattice in earnest use)
        _lattice("slab_64_f64", 64, 64, "fp64", "bgk", "guo", "slab", 0.8, 1.0, -0.304, 1.0, 200, 16.0, out="moments", source="host"),
        # a static droplet of the temperature and relaxation-time sweep, FP64 and FP32 deviations
        _lattice("droplet_256_f64", 256, 256, "fp64", "mrt", "guo", "droplet", 0.7, 0.8, -0.84, 0.25, 50, 40.0),
        _lattice("droplet_256_f32", 256, 256, "fp32", "mrt", "guo", "droplet", 0.7, 0.8, -0.84, 0.25, 200, 40.0),
        # the FP64 step at a size that fills the GPU
        _lattice("array_1024_f64", 1024, 1024, "fp64", "mrt", "guo", "array", 0.7, 0.8, -0.304, 1.0, 10, 80.0, cell=256),
        # a box whose sides are no multiple of four, nor of a tile
        _lattice("ragged_1023_f32", 1023, 1021, "fp32", "bgk", "guo", "droplet", 0.8, 0.9, -0.304, 1.0, 50, 250.0),
        # the throughput case: 16 x 16 droplets on 4096 x 4096
        _lattice("array_4096_f32", 4096, 4096, "fp32", "mrt", "guo", "array", 0.7, 0.8, -0.304, 1.0, 20, 80.0, cell=256),
        # one convergence check of that case: observables, comparison with the last snapshot, new snapshot
        dict(kind="stats", name="stats_4096_f32", nx=4096, ny=4096, precision="fp32", collision="mrt", forcing="guo", field="array",
             T=0.7, tau=0.8, A=-0.304, K=1.0, size=80.0, cell=256),
        # the start of a large run
        dict(kind="preset", name="preset_2048_f32", nx=2048, ny=2048, precision="fp32", field="droplet_array", T=0.7, tau=0.8, A=-0.304,
             K=1.0, size=80.0, cell=256),
        # a flat-interface temperature grid: many narrow slabs at once
        dict(kind="batch", name="batch_slabs", n=24, shapes="8x128", collision="bgk", forcing="guo", steps=200, pick=1, profiles=False),
        # the droplet and slab sweep with uneven sides (half of the 512 instances), profiles out as the warm start's training set
        dict(kind="batch", name="batch_sweep", n=256, shapes="sweep", collision="mrt", forcing="guo", steps=30, pick=2, profiles=True),
        # two passes over the 2000 converged profiles in minibatches of 64
        dict(kind="train", name="net_train", n=2000, epochs=2, batch=64),
        # the held-out sweep's profiles
        dict(kind="predict", name="net_predict", n=256),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    what = rng.choice(["lattice", "lattice", "lattice", "lattice", "stats", "preset", "batch", "batch", "train", "predict"])
    if what in ("train", "predict"):
        n = _log(rng, 30, 2500)
        return dict(kind="predict", n=n) if what == "predict" else dict(kind="train", n=n, epochs=rng.randint(1, 2), batch=rng.choice([32, 50, 64, 100, 256]))
    collision, forcing = rng.choice([("bgk", "guo"), ("bgk", "edm"), ("bgk", "sc"), ("bgk", "li"), ("mrt", "guo"), ("mrt", "guo")])
    if what == "batch":
        if rng.random() < 0.4:
            return dict(kind="batch", n=rng.randint(3, 60), shapes="8x%d" % rng.choice([63, 96, 127, 128, 200]), collision=collision,
                        forcing=forcing, steps=rng.randint(50, 200), pick=rng.randint(1, 10 ** 6), profiles=False)
        return dict(kind="batch", n=_log(rng, 2, 256), shapes="sweep", collision="mrt", forcing="guo", steps=rng.randint(10, 25),
                    pick=rng.randint(1, 10 ** 6), profiles=rng.random() < 0.5)
    precision = rng.choice(["fp32", "fp32", "fp64"]) if what == "lattice" else "fp32"
    top = 1024 if precision == "fp64" else 4096
    nx, ny = _log(rng, 48, top), _log(rng, 48, top)
    if rng.random() < 0.65:
        nx = max(48, nx // 4 * 4)
    side = min(nx, ny)
    T = rng.choice([0.7, 0.8, 0.9])
    c = dict(kind=what, nx=nx, ny=ny, precision=precision, field="droplet_array" if what == "preset" else "droplet", T=T,
             tau=round(rng.uniform(0.7, 1.2), 2), A=-0.304, K=1.0, size=round(side * rng.uniform(0.2, 0.3), 1), cell=side)
    if what == "preset":
        return c
    c.update(collision=collision, forcing=forcing, A=0.0 if forcing == "li" else -0.84)
    if what == "stats":
        return c
    nodes = nx * ny
    steps = max(5, min(200, int((4e6 if precision == "fp64" else 6e7) / nodes)))
    c.update(steps=steps, source=rng.choice(["host", "device"]) if nodes < 3e5 else "device", out="moments" if precision == "fp64" and rng.random() < 0.5 else "state")
    return c


# ---- inputs ----

def _coexistence(T):
    """Coexistence densities of the EOS at T/Tc (equal pressure and chemical potential), by Newton's method in (log rho_v, rho_l)."""
    t = T * TC
    at = [(0.5, -6.72, 0.4534), (0.6, -5.78, 0.4062), (0.7, -4.69, 0.358), (0.8, -3.92, 0.307), (0.9, -3.2, 0.245)]
    x = np.array([np.interp(T, [a[0] for a in at], [a[k] for a in at]) for k in (1, 2)])

    def mu_p(r):
        ex, dex = (4 * r - 3 * r * r) / (1 - r) ** 2, (4 - 2 * r) / (1 - r) ** 3
        f = r * t * math.log(r) + r * t * ex - r * r
        mu = t * (math.log(r) + 1) + t * (ex + r * dex) - 2 * r
        return mu, r * mu - f

    def res(v):
        a, b = mu_p(math.exp(v[0])), mu_p(v[1])
        return np.array([a[0] - b[0], (a[1] - b[1]) * 100])

    for _ in range(60):
        r, h = res(x), 1e-7
        J = np.stack([(res(x + np.eye(2)[k] * h) - res(x - np.eye(2)[k] * h)) / (2 * h) for k in (0, 1)], 1)
        d = np.linalg.solve(J, -r)
        x = x + d * min(1.0, 0.3 / (abs(d[0]) + 1e-300), 0.02 / (abs(d[1]) + 1e-300))
    return math.exp(x[0]), float(x[1])


def _vapour(T):
    """The reference density of FP32 deviations: the vapour density, a float."""
    return float(np.float32(_coexistence(T)[0]))


def _field(c, seed):
    """Initial density on the device: tanh interfaces of width 4 with 1e-6 noise, the liquid's place and size moved a little by the seed."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    j = np.random.RandomState(seed).uniform(-1, 1, 3)
    rv, rl = _coexistence(c["T"])
    y = torch.arange(c["ny"], device="cuda", dtype=torch.float64)[:, None]
    x = torch.arange(c["nx"], device="cuda", dtype=torch.float64)[None, :]
    cx, cy, size = c["nx"] / 2 + j[0], c["ny"] / 2 + j[1], c["size"] + 0.5 * j[2]
    if c["field"] == "slab":
        d = (y - cy).abs() - size + 0.5 * torch.cos(2 * math.pi * x / c["nx"] + j[0])
    elif c["field"] == "array":
        d = torch.hypot(x - torch.floor(x / c["cell"]) * c["cell"] - c["cell"] / 2 - j[0], y - torch.floor(y / c["cell"]) * c["cell"] - c["cell"] / 2 - j[1]) - size
    else:
        d = torch.hypot(x - cx, y - cy) - size
    noise = 2 * torch.rand(c["ny"], c["nx"], device="cuda", dtype=torch.float64, generator=g) - 1
    return (rv + (rl - rv) * 0.5 * (1 - torch.tanh(d / 2)) + 1e-6 * noise).contiguous()


def _params(c):
    return lbm.make_params(c["nx"], c["ny"], c["T"], c["tau"], c["A"], c["K"], c.get("collision", "mrt"), c.get("forcing", "guo"), c["precision"],
                           rho_ref=_vapour(c["T"]) if c["precision"] == "fp32" else 0.0, sigma=0.105 if c.get("forcing") == "li" else 0.0, **RATES)


def _instances(c, seed):
    """A batch's instances: the sides from the case alone, everything else from the seed."""
    pick, r = np.random.RandomState(c["pick"]), np.random.RandomState(seed)
    out = []
    for i in range(c["n"]):
        if c["shapes"] == "sweep":
            nx = ny = int(pick.choice(np.arange(64, 513, 32)))
            T, tau, K, kind, size = r.uniform(0.5, 0.9), r.uniform(0.55, 1.2), r.uniform(1 / 16, 1), "droplet" if pick.rand() < 0.5 else "slab", r.uniform(10, max(11, nx / 4))
        else:
            nx, ny = (int(v) for v in c["shapes"].split("x"))
            T, tau, K, kind, size = 0.7 + 0.2 * (i % 8) / 8 + r.uniform(0, 0.02), r.uniform(0.8, 1.2), 1.0, "slab", ny / 4
        rv, rl = _coexistence(T)
        A = 0.0 if c["forcing"] == "li" else -0.84
        out.append(dict(nx=nx, ny=ny, kind=kind, T_over_Tc=T, tau=tau, A=A, K=K, size=size, rho_l=rl, rho_v=rv, seed=seed * 1000 + i, noise_amp=1e-6))
    return out


def _grid(inst):
    """Sample grid of an instance's profile: centred on its interface, half a lattice unit apart at K = 1."""
    return [(1, d["size"], 0.5 / math.sqrt(d["K"])) for d in inst]


def _net_inputs(c, seed):
    """Rows (T/Tc, tau, A, K, radius) of a sweep and log-density-like profiles across an interface, with their scalings and initial weights."""
    r = np.random.RandomState(seed)
    X = r.uniform([0.5, 0.55, -0.84, 1 / 16, 10], [0.9, 1.2, -0.83999, 1.0, 128], (c["n"], 5)).astype(np.float32)
    s = (np.arange(SAMPLES) - (SAMPLES - 1) / 2) / 8
    wide = 0.6 + 1.5 * X[:, :1] + 0.2 * X[:, 3:4]
    Y = (1.02 - 0.1 * X[:, 1:2] - (1 + 0.05 * X[:, :1]) * 0.5 * (1 + np.tanh(s[None, :] / wide - 2 / X[:, 4:5])) + 1e-3 * r.randn(c["n"], SAMPLES)).astype(np.float32)
    theta = np.concatenate([v for i, o in zip(NET, NET[1:]) for v in (r.uniform(-1, 1, o * i) * math.sqrt(6 / (i + o)), np.zeros(o))]).astype(np.float32)
    xs = X.std(0)
    xs[2] = 1
    return X, Y, theta, (X.mean(0), xs, Y.mean(0), Y.std(0) + np.float32(1e-3))


# ---- what a program has in hand, and one pass ----

def prepare(case, seed):
    c, k = case, case["kind"]
    if k in ("train", "predict"):
        X, Y, theta, scale = _net_inputs(c, seed)
        net = lbm.WarmStartNet(seed=0)
        net.set_scaling(*scale)
        net.set_params(theta)
        return dict(case=c, net=net, X=X, Y=Y, theta=theta, seed=seed)
    if k == "batch":
        inst = _instances(c, seed)
        return dict(case=c, batch=lbm.Batch(inst, c["collision"], c["forcing"], sigma=0.105 if c["forcing"] == "li" else 0.0, **RATES), grid=_grid(inst))
    lat = lbm.Lattice(_params(c))
    s = dict(case=c, lat=lat, seed=seed)
    if k != "preset":
        rho0 = _field(c, seed)
        s["rho0"] = rho0.cpu().numpy() if c.get("source") == "host" else rho0
    if k == "stats":
        torch.cuda.synchronize()
        lat.init_density_dev(s["rho0"])
        lat.stats(snapshot=True)
        lat.step(2)
    elif c.get("out") != "moments":
        s["state"] = torch.empty(9, c["ny"], c["nx"], dtype=torch.float64 if c["precision"] == "fp64" else torch.float32, device="cuda")
    torch.cuda.synchronize()
    return s


def run(state):
    s, c = state, state["case"]
    k = c["kind"]
    if k == "train":
        s["net"].set_params(s["theta"])
        loss = s["net"].train(s["X"], s["Y"], c["epochs"], c["batch"], lr=2e-3, seed=s["seed"])
        return dict(loss=loss, params=s["net"].get_params())
    if k == "predict":
        return s["net"].predict(s["X"])
    if k == "batch":
        b = s["batch"]
        b.init()
        b.step(c["steps"])
        b.observe()
        state_, code, steps, obs = b.results()
        # the batch's populations and arithmetic are FP32: its observables and profiles are kept as such
        out = dict(state=state_, code=code, steps=steps, obs={n: v.astype(np.float32) for n, v in obs.items()})
        if c["profiles"]:
            out["profiles"] = b.profiles(SAMPLES, s["grid"]).astype(np.float32)
        return out
    lat = s["lat"]
    if k == "stats":
        return lat.stats(snapshot=True)
    if k == "preset":
        rv, rl = _coexistence(c["T"])
        lat.init_preset(c["field"], c["size"], rho_l=rl, rho_v=rv, cell=c["cell"], seed=s["seed"])
        st = lat.stats()
        lat.copy_rows(0, s["state"])
        return dict(stats=st, state=s["state"])
    if c["source"] == "host":
        lat.init_density(s["rho0"])
    else:
        lat.init_density_dev(s["rho0"])
    lat.step(c["steps"])
    if c["out"] == "moments":
        return lat.read_moments()
    lat.copy_rows(0, s["state"])
    return s["state"]


def work(case):
    """One pass: every population read and written once a step (observables: read once), the model's operations per node."""
    c, k = case, case["kind"]
    if k in ("train", "predict"):
        p = sum(a * b + b for a, b in zip(NET, NET[1:]))
        if k == "predict":
            return dict(bytes=4 * (p + c["n"] * (NET[0] + NET[-1])), flops=2 * p * c["n"])
        updates = c["epochs"] * -(-c["n"] // c["batch"])
        return dict(bytes=4 * c["epochs"] * c["n"] * (NET[0] + NET[-1]) + 24 * p * updates, flops=6 * p * c["n"] * c["epochs"] + 2 * p * c["n"])
    if k == "batch":
        nodes = sum(d["nx"] * d["ny"] for d in _instances(c, 1))
        return dict(bytes=nodes * (72 * c["steps"] + 36 + 36), flops=nodes * 260 * c["steps"])
    nodes, b = c["nx"] * c["ny"], 8 if c["precision"] == "fp64" else 4
    if k == "stats":
        return dict(bytes=nodes * (9 * b + 4 * b), flops=nodes * 120)
    if k == "preset":
        return dict(bytes=nodes * 9 * b * 4, flops=nodes * 200)
    return dict(bytes=nodes * (18 * b * c["steps"] + 8 + 9 * b + (24 if c["out"] == "moments" else 18 * b)), flops=nodes * 260 * c["steps"])


# ---- the same in 64 bits ----

class _Model:
    """The update of B lattices of one shape, (9, B, ny, nx) stored populations f*_a(x, t-1) pulled by the next step."""

    def __init__(self, T, tau, A, K, collision, forcing):
        t = lambda v: torch.tensor(v, dtype=torch.float64, device="cuda").reshape(-1, 1, 1)  # noqa: E731
        self.T, self.tau, self.A, self.K = t([x * TC for x in T]), t(tau), t(A), t(K)
        self.collision, self.forcing = collision, forcing

    def start(self, rho0):
        return torch.stack([w * torch.roll(rho0, (-ey, -ex), (1, 2)) for w, (ex, ey) in zip(W, E)])

    def macro(self, s):
        f = torch.stack([torch.roll(s[a], (ey, ex), (1, 2)) for a, (ex, ey) in enumerate(E)])
        rho = f.sum(0)
        jx, jy = (sum(e[k] * f[a] for a, e in enumerate(E) if e[k]) for k in (0, 1))
        p = self.K * (rho * self.T * (1 + rho + rho ** 2 - rho ** 3) / (1 - rho) ** 3 - rho ** 2)
        psi = (2 * (rho / 3 - p)).sqrt()
        Fx, Fy = torch.zeros_like(rho), torch.zeros_like(rho)
        for ex, ey in E[1:]:
            n = torch.roll(psi, (-ey, -ex), (1, 2))
            phi = (1 / 3 if ex * ey == 0 else 1 / 12) * n * (self.A / 2 * n + (1 - self.A) * psi)
            Fx, Fy = Fx + ex * phi, Fy + ey * phi
        return f, rho, jx / rho, jy / rho, Fx, Fy, psi

    def velocity(self, s):
        _, rho, ux, uy, Fx, Fy, _ = self.macro(s)
        return rho, ux + Fx / (2 * rho), uy + Fy / (2 * rho)

    def step(self, s):
        f, rho, ux, uy, Fx, Fy, psi = self.macro(s)
        vx, vy = ux + Fx / (2 * rho), uy + Fy / (2 * rho)

        def feq(x, y):
            q = 1.5 * (x * x + y * y)
            return torch.stack([w * rho * (1 + 3 * (ex * x + ey * y) + 4.5 * (ex * x + ey * y) ** 2 - q) for w, (ex, ey) in zip(W, E)])

        def source(x, y):
            d = 3 * (x * Fx + y * Fy)
            return torch.stack([w * ((ex * Fx + ey * Fy) * (3 + 9 * (ex * x + ey * y)) - d) for w, (ex, ey) in zip(W, E)])

        if self.collision == "mrt":
            e2 = [ex * ex + ey * ey for ex, ey in E]
            M = torch.tensor([[1.0] * 9, [-4 + 3 * q for q in e2], [4 - 10.5 * q + 4.5 * q * q for q in e2], [e[0] for e in E], [(3 * q - 5) * e[0] for q, e in zip(e2, E)],
                              [e[1] for e in E], [(3 * q - 5) * e[1] for q, e in zip(e2, E)], [e[0] ** 2 - e[1] ** 2 for e in E], [e[0] * e[1] for e in E]], dtype=torch.float64, device=s.device)
            r = torch.ones(9, len(self.tau), 1, 1, dtype=torch.float64, device=s.device)
            r[1], r[2], r[4], r[6], r[7], r[8] = RATES["s_e"], RATES["s_eps"], RATES["s_q"], RATES["s_q"], 1 / self.tau, 1 / self.tau
            m = torch.tensordot(M, f, 1)
            m = m - r * (m - torch.tensordot(M, feq(vx, vy), 1)) + (1 - r / 2) * torch.tensordot(M, source(vx, vy), 1)
            return torch.tensordot(M.T / (M * M).sum(1), m, 1)
        if self.forcing == "edm":
            q = feq(ux, uy)
            return f + (q - f) / self.tau + feq(ux + Fx / rho, uy + Fy / rho) - q
        if self.forcing == "sc":
            return f + (feq(ux + self.tau * Fx / rho, uy + self.tau * Fy / rho) - f) / self.tau
        h = 0.105 / ((self.tau - 0.5) * psi * psi) if self.forcing == "li" else 0.0
        return f + (feq(vx, vy) - f) / self.tau + (1 - 0.5 / self.tau) * source(vx + h * Fx, vy + h * Fy)


def _observables(model, s, before=None):
    """lbm_stats' fields, and a batch's, of every lattice."""
    rho, vx, vy = model.velocity(s)
    ny, nx = rho.shape[1:]
    o = dict(mass=rho.sum((1, 2)), max_v=torch.hypot(vx, vy).amax((1, 2)), rho_min=rho.amin((1, 2)), rho_max=rho.amax((1, 2)), rho_center=rho[:, ny // 2, nx // 2],
             rho_corner=rho[:, 0, 0], rho_row_mid=rho[:, ny // 2].mean(1), rho_row0=rho[:, 0].mean(1))
    if before is not None:
        o["max_dv"] = torch.hypot(vx - before[0], vy - before[1]).amax((1, 2))
    return o, rho


def _one(c):
    return _Model([c["T"]], [c["tau"]], [c["A"]], [c["K"]], c.get("collision", "mrt"), c.get("forcing", "guo"))


def _stored(c, s):
    ref = _vapour(c["T"]) if c["precision"] == "fp32" else 0.0
    return torch.stack([s[a, 0] - W[a] * ref for a in range(9)])


def _noise(nx, ny, seed):
    """2 xi - 1 of the presets' noise, xi from SplitMix64 of seed ^ node."""
    with np.errstate(over="ignore"):
        z = (np.uint64(seed) ^ np.arange(nx * ny, dtype=np.uint64)) + np.uint64(0x9E3779B97F4A7C15)
        z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
        z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
        z = (z ^ (z >> np.uint64(31))) >> np.uint64(11)
    return torch.from_numpy(2 * (z.astype(np.float64) / 2.0 ** 53) - 1).cuda().reshape(ny, nx)


def _preset(nx, ny, kind, size, cell, rv, rl, seed):
    y = torch.arange(ny, device="cuda", dtype=torch.float64)[:, None]
    x = torch.arange(nx, device="cuda", dtype=torch.float64)[None, :]
    if kind == "slab":
        d = (y - ny / 2).abs() - size + 0 * x
    elif kind == "droplet_array":
        d = torch.hypot(x - torch.floor(x / cell) * cell - cell / 2, y - torch.floor(y / cell) * cell - cell / 2) - size
    else:
        d = torch.hypot(x - nx / 2, y - ny / 2) - size
    return rv + (rl - rv) * 0.5 * (1 - torch.tanh(d / 2)) + 1e-6 * _noise(nx, ny, seed)


def _profile(rho, kind, centre, spacing):
    """Mean density over 64 directions (slab: both sides of the mid-row) at the sample radii, bilinear between nodes."""
    ny, nx = rho.shape
    far = (ny if kind == "slab" else min(nx, ny)) / 2 - 1
    r = (centre + spacing * (torch.arange(SAMPLES, device="cuda", dtype=torch.float64) - (SAMPLES - 1) / 2)).abs().clamp(max=far)
    if kind == "slab":
        row = rho.mean(1)
        yy = torch.stack([ny / 2 - r, ny / 2 + r])
        y0 = torch.floor(yy)
        t, k = yy - y0, y0.long()
        return ((1 - t) * row[k % ny] + t * row[(k + 1) % ny]).mean(0)
    th = 2 * math.pi * torch.arange(64, device="cuda", dtype=torch.float64)[:, None] / 64
    xx, yy = nx / 2 + r * torch.cos(th), ny / 2 + r * torch.sin(th)
    x0, y0 = torch.floor(xx), torch.floor(yy)
    tx, ty, i, j = xx - x0, yy - y0, x0.long(), y0.long()
    at = lambda dy, dx: rho[(j + dy) % ny, (i + dx) % nx]  # noqa: E731
    return ((1 - ty) * ((1 - tx) * at(0, 0) + tx * at(0, 1)) + ty * ((1 - tx) * at(1, 0) + tx * at(1, 1))).mean(0)


def _exact_batch(c, seed):
    inst = _instances(c, seed)
    obs, prof = {n: np.zeros(c["n"]) for n in lbm.BATCH_OBS}, np.zeros((c["n"], SAMPLES))
    for shape in sorted({(d["ny"], d["nx"]) for d in inst}):
        ids = [i for i, d in enumerate(inst) if (d["ny"], d["nx"]) == shape]
        some = [inst[i] for i in ids]
        m = _Model([d["T_over_Tc"] for d in some], [d["tau"] for d in some], [d["A"] for d in some], [d["K"] for d in some], c["collision"], c["forcing"])
        s = m.start(torch.stack([_preset(d["nx"], d["ny"], d["kind"], d["size"], 0, d["rho_v"], d["rho_l"], d["seed"]) for d in some]))
        for _ in range(c["steps"]):
            s = m.step(s)
        o, rho = _observables(m, s)
        for n, v in o.items():
            obs[n][ids] = v.cpu().numpy()
        for k, i in enumerate(ids):
            prof[i] = _profile(rho[k], inst[i]["kind"], *_grid([inst[i]])[0][1:]).cpu().numpy()
    obs["max_dv"] = obs["max_drho"] = None     # no earlier check to compare with
    return dict(dict(state=None, code=None, steps=None, obs=obs), **({"profiles": prof} if c["profiles"] else {}))


def _shuffle(n, seed, epoch):
    """Fisher-Yates on SplitMix64 draws, as lbm_ws_train documents its per-epoch order."""
    mask = (1 << 64) - 1
    perm = list(range(n))
    for i in range(n - 1, 0, -1):
        z = ((seed ^ (epoch << 32) ^ i) + 0x9E3779B97F4A7C15) & mask
        z = ((z ^ (z >> 30)) * 0xBF58476D1CE4E5B9) & mask
        z = ((z ^ (z >> 27)) * 0x94D049BB133111EB) & mask
        j = (z ^ (z >> 31)) % (i + 1)
        perm[i], perm[j] = perm[j], perm[i]
    return perm


def _exact_net(c, seed):
    X, Y, theta, scale = _net_inputs(c, seed)
    X, Y, theta, xm, xs, ym, ys = (torch.tensor(v, dtype=torch.float64, device="cuda") for v in (X, Y, theta, *scale))
    p = theta.clone().requires_grad_(True)

    def forward(x):
        h, o = (x - xm) / xs, 0
        for k, (i, n) in enumerate(zip(NET, NET[1:])):
            h = h @ p[o:o + n * i].reshape(n, i).T + p[o + n * i:o + n * i + n]
            o += n * i + n
            h = torch.tanh(h) if k < len(NET) - 2 else h
        return h

    if c["kind"] == "predict":
        with torch.no_grad():
            return (forward(X) * ys + ym).cpu().numpy()
    opt = torch.optim.Adam([p], lr=2e-3, betas=(0.9, 0.999), eps=1e-8)
    for ep in range(c["epochs"]):
        order = torch.tensor(_shuffle(c["n"], seed, ep), device="cuda")
        for at in range(0, c["n"], min(c["batch"], c["n"])):
            k = order[at:at + min(c["batch"], c["n"])]
            opt.zero_grad()
            ((forward(X[k]) - (Y[k] - ym) / ys) ** 2).mean().backward()
            opt.step()
    with torch.no_grad():
        loss = float(((forward(X) - (Y - ym) / ys) ** 2).mean())
    return dict(loss=loss, params=p.detach().cpu().numpy())


def exact(case, seed):
    c, k = case, case["kind"]
    if k in ("train", "predict"):
        return _exact_net(c, seed)
    if k == "batch":
        return _exact_batch(c, seed)
    m = _one(c)
    if k == "preset":
        rv, rl = _coexistence(c["T"])
        s = m.start(_preset(c["nx"], c["ny"], "droplet_array", c["size"], c["cell"], rv, rl, seed)[None])
        o, _ = _observables(m, s)
        return dict(stats=dict({n: float(v) for n, v in o.items()}, max_dv=None, steps=None, status=None), state=_stored(c, s))
    s = m.start(_field(c, seed)[None])
    if k == "stats":
        before = m.velocity(s)[1:]
        for _ in range(2):
            s = m.step(s)
        return dict({n: float(v) for n, v in _observables(m, s, before)[0].items()}, steps=None, status=None)
    for _ in range(c["steps"]):
        s = m.step(s)
    if c["out"] == "moments":
        return tuple(v[0].cpu().numpy() for v in m.velocity(s))
    return _stored(c, s)
