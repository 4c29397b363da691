"""What this framework is used for, as cases that can be timed and compared.

A case is a plain dict; `prepare` makes what a user's program has in hand (fields on the GPU or
on the host, a lattice, batch or network handle), `run` is one pass through the public entry
points, `exact` the same pass in plain 64-bit torch.  A lattice's pass starts the state from its
fields, takes the steps between two checks of a run (100, the library's own cadence, unless the
case says otherwise) and reads the density and velocity fields.
"""
import math

import numpy as np
import torch

A_EOS, B_EOS, SIGMA, G = 0.25, 4.0, 0.114, -1.0
RATES = (1.0, 1.1, 1.1, 1.0, 1.1, 1.0, 1.1, 1.0, 1.0)
SPLASH_RATES = (1.0, 0.8, 0.8, 1.0, 1.1, 1.0, 1.1, 1.0, 1.0)
WIDTH = 4.0
ADAM = dict(lr=1e-3, beta1=0.9, beta2=0.999, eps=1e-8)


def listed():
    return [
        # A narrow flat film, the smallest lattice of the coexistence and calibration sweeps:
        # launches and latency are all there is.
        lattice("film_64x64", 64, 64, "film", visc="const", tr=0.7, steps=100),
        # The stationary droplet of the paper in double precision (Laplace's law, spurious
        # currents): a small grid in the parity mode.
        lattice("droplet_128x128_fp64", 128, 128, "droplet", "fp64", "const", 0.7, 100),
        # One droplet on an odd, ragged grid with a viscosity step, in single precision: the
        # size of most members of a parameter study.
        lattice("droplet_193x147", 193, 147, "droplet", visc="step", tr=0.8, steps=100),
        # A host program without a GPU array library: double fields in and out of host memory.
        lattice("droplet_601x407_host", 601, 407, "droplet", visc="linear", tr=0.7, steps=100,
                io="host"),
        # The oscillating ellipse, the accuracy workload of the FP32 mode.
        lattice("ellipse_1024x1024", 1024, 1024, "ellipse", visc="linear", tr=0.6, steps=100),
        # The splash on a thin film between walls, with moving liquid.
        lattice("splash_2048x512", 2048, 512, "splash", visc="step", tr=0.5, steps=100,
                bc="walls"),
        # FP32 storage with psi evaluated in double (the option for low reduced temperatures),
        # on a size that is no multiple of a tile.
        lattice("droplets_1300x900_psi64", 1300, 900, "droplets", visc="linear", tr=0.6,
                steps=50, psi_fp64=True),
        # The double-precision parity run of a mid-sized field.
        lattice("droplets_1024x1024_fp64", 1024, 1024, "droplets", "fp64", "linear", 0.7, 20),
        # The throughput workload: 64 droplets on 4096 x 4096, far larger than the L2 cache.
        lattice("droplets_4096x4096", 4096, 4096, "droplets", visc="linear", tr=0.7, steps=100),
        # The batched equilibria that make the network's training data: films and droplets of
        # 256 ragged sizes and parameters, stepped with a convergence check every 100 steps.
        {"name": "batch_256", "kind": "batch", "n": 256, "lo": 64, "hi": 512, "steps": 600},
        # Training of the warm-start network on such data: 256 rows, a fifth of an epoch count.
        {"name": "train_256", "kind": "train", "rows": 256, "updates": 200},
        # A warm-started field of 64 droplets (balanced velocities, curvature-corrected
        # densities) up to its first convergence check.
        {"name": "warm_4096x4096", "kind": "warm", "nx": 4096, "ny": 4096, "drops": 64,
         "tr": 0.7, "steps": 100},
    ]


def lattice(name, nx, ny, shape, precision="fp32", visc="const", tr=0.7, steps=100,
            bc="periodic", psi_fp64=False, io="device"):
    case = {"name": name, "kind": "lattice", "nx": nx, "ny": ny, "shape": shape,
            "precision": precision, "visc": visc, "tr": tr, "steps": steps, "bc": bc,
            "psi_fp64": psi_fp64, "io": io}
    return case


def draw(rng):
    """One more case of the same ranges: mostly single lattices of any size and option."""
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    p = rng.random()
    if p < 0.1:
        lo = log_int(48, 96)
        return {"kind": "batch", "n": log_int(8, 200), "lo": lo, "hi": log_int(128, 500),
                "steps": rng.choice([200, 300, 500])}
    if p < 0.15:
        return {"kind": "train", "rows": log_int(32, 256), "updates": rng.randrange(50, 201)}
    if p < 0.2:
        return {"kind": "warm", "nx": log_int(512, 3000), "ny": log_int(512, 3000),
                "drops": log_int(4, 24), "tr": round(rng.uniform(0.6, 0.8), 3),
                "steps": rng.choice([50, 100])}
    fp64 = rng.random() < 0.25
    hi = 1000 if fp64 else 4000
    case = lattice("", log_int(60, hi), log_int(60, hi),
                   rng.choice(["film", "droplet", "ellipse", "splash", "droplets"]),
                   "fp64" if fp64 else "fp32", rng.choice(["const", "step", "linear"]),
                   round(rng.uniform(0.55, 0.85), 3), 100,
                   rng.choice(["periodic", "periodic", "walls"]),
                   not fp64 and rng.random() < 0.15,
                   "host" if rng.random() < 0.15 else "device")
    if case["shape"] == "splash":
        case["bc"] = "walls"
    if fp64:
        case["steps"] = rng.choice([10, 20]) if case["nx"] * case["ny"] > 1 << 16 else 100
    elif case["psi_fp64"]:
        case["steps"] = 50
    else:
        case["steps"] = rng.choice([50, 64, 100, 100, 128])
    if case["io"] == "host" and case["nx"] * case["ny"] > 1 << 20:
        case["io"] = "device"
    del case["name"]
    return case


# ---------------------------------------------------------------------------------------
# Equation of state: Carnahan-Starling with a, b and R = 1, at T = tr * 0.3773 a / b.
def temperature(tr, a=A_EOS):
    return tr * 0.3773 * a / B_EOS


def _p(r, a, T):
    x = 0.25 * B_EOS * r
    return r * T * (1 + x + x * x - x ** 3) / (1 - x) ** 3 - a * r * r


def _mu(r, a, T):
    """Chemical potential up to a constant: p / r + the integral of p / r^2."""
    x = 0.25 * B_EOS * r
    return T * (np.log(r) + (4 * x - 3 * x * x) / (1 - x) ** 2) - a * r + _p(r, a, T) / r


def _bisect(f, lo, hi):
    """Element-wise root of f, which changes sign between lo and hi."""
    up = f(hi) > 0
    for _ in range(60):
        mid = 0.5 * (lo + hi)
        right = (f(mid) > 0) == up
        lo, hi = np.where(right, lo, mid), np.where(right, mid, hi)
    return 0.5 * (lo + hi)


def coexistences(a, T):
    """(rho_l, rho_v) of equal pressure and chemical potential, for arrays of a and T."""
    a, T = np.asarray(a, dtype=np.float64), np.asarray(T, dtype=np.float64)
    rs = np.linspace(1e-6, 4.0 / B_EOS * 0.75, 4001)
    falling = np.diff(_p(rs, a[:, None], T[:, None]), axis=1) < 0
    s1 = rs[np.argmax(falling, axis=1)]  # spinodals, to a step of the table
    s2 = rs[falling.shape[1] - np.argmax(falling[:, ::-1], axis=1)]

    def pair(p0):
        return (_bisect(lambda r: _p(r, a, T) - p0, s2, np.full_like(s2, 4.0 / B_EOS * 0.999)),
                _bisect(lambda r: _p(r, a, T) - p0, np.full_like(s1, 1e-12), s1))

    def gap(p0):
        rl, rv = pair(p0)
        return _mu(rl, a, T) - _mu(rv, a, T)

    lo = np.maximum(_p(s2, a, T), 1e-12)
    return pair(_bisect(gap, lo * (1 + 1e-9), _p(s1, a, T) * (1 - 1e-9)))


def coexistence(a, T):
    rl, rv = coexistences([a], [T])
    return float(rl[0]), float(rv[0])


# ---------------------------------------------------------------------------------------
# Inputs, from the seed alone.
def _profile(d, rl, rv):
    return 0.5 * (rl + rv) - 0.5 * (rl - rv) * torch.tanh(2.0 * d / WIDTH)


def _layout(nx, ny, n, rng):
    """Centres and radii of up to n droplets that do not touch (periodic)."""
    rmax = min(0.35 * min(nx, ny), max(10.0, 0.62 * math.sqrt(nx * ny / n) / 2))
    drops, tries = [], 0
    while len(drops) < n and tries < 400 * n:
        tries += 1
        r = rng.uniform(0.35 * rmax, rmax)
        cx, cy = rng.uniform(0, nx), rng.uniform(0, ny)
        if all(math.hypot(min(abs(cx - x), nx - abs(cx - x)), min(abs(cy - y), ny - abs(cy - y)))
               > r + q + 3 * WIDTH for x, y, q in drops):
            drops.append((cx, cy, r))
    return np.array(drops)


def _drops_field(nx, ny, drops, rl, rv, shift=0.0, width=WIDTH):
    """The largest over the droplets of the tanh profile about each one's circle."""
    rho = torch.full((ny, nx), rv, dtype=torch.float64, device="cuda")
    for cx, cy, r in drops:
        reach = int(r + 9 * width) + 2
        xs = torch.arange(int(cx) - reach, int(cx) + reach + 1, device="cuda")[:nx]
        ys = torch.arange(int(cy) - reach, int(cy) + reach + 1, device="cuda")[:ny]
        dx = torch.abs(torch.remainder(xs, nx).double() - cx)
        dy = torch.abs(torch.remainder(ys, ny).double() - cy)
        dx, dy = torch.minimum(dx, nx - dx), torch.minimum(dy, ny - dy)
        d = torch.sqrt(dx[None, :] ** 2 + dy[:, None] ** 2) - (r + shift)
        v = 0.5 * (rl + rv) - 0.5 * (rl - rv) * torch.tanh(2.0 * d / width)
        at = (torch.remainder(ys, ny)[:, None], torch.remainder(xs, nx)[None, :])
        rho[at] = torch.maximum(rho[at], v)
    return rho


def _fields(case, seed):
    """rho, ux, uy (ny, nx) doubles on the GPU; the velocities are None for a start at rest."""
    nx, ny = case["nx"], case["ny"]
    rl, rv = coexistence(A_EOS, temperature(case["tr"]))
    rng = np.random.default_rng(seed)
    y, x = torch.meshgrid(torch.arange(ny, device="cuda").double(),
                          torch.arange(nx, device="cuda").double(), indexing="ij")
    cx, cy = (nx - 1) / 2.0 + rng.uniform(-2, 2), (ny - 1) / 2.0 + rng.uniform(-2, 2)
    size = min(nx, ny)
    ux = uy = None
    if case["shape"] == "film":
        rho = _profile(torch.abs(y - cy) - ny * rng.uniform(0.22, 0.28), rl, rv)
    elif case["shape"] == "droplet":
        rho = _profile(torch.hypot(x - cx, y - cy) - size * rng.uniform(0.22, 0.26), rl, rv)
    elif case["shape"] == "ellipse":
        th = torch.atan2(y - cy, x - cx)
        ea, eb = nx * 0.234, ny * rng.uniform(0.15, 0.16)
        re = ea * eb / torch.sqrt((eb * torch.cos(th)) ** 2 + (ea * torch.sin(th)) ** 2)
        rho = _profile(torch.hypot(x - cx, y - cy) - re, rl, rv)
    elif case["shape"] == "splash":
        film, dia = 0.0625 * ny, 0.31 * size * rng.uniform(0.95, 1.05)
        drop = _profile(torch.hypot(x - cx, y - (film + dia / 2 + 2 * WIDTH)) - dia / 2, rl, rv)
        rho = torch.maximum(_profile(y - (film - 0.5), rl, rv), drop)
        ux = torch.zeros_like(rho)
        uy = -0.05 * torch.clamp((drop - rv) / (rl - rv), 0.0, 1.0)
    else:
        n = max(2, min(64, nx * ny // 40000))
        rho = _drops_field(nx, ny, _layout(nx, ny, n, rng), rl, rv)
    gen = torch.Generator(device="cuda").manual_seed(int(seed))
    noise = torch.rand(rho.shape, generator=gen, device="cuda", dtype=torch.float64)
    rho = rho * (1.0 + 1e-4 * (2.0 * noise - 1.0))
    return rho, ux, uy, rl, rv


def _rates(case):
    return SPLASH_RATES if case["shape"] == "splash" else RATES


def _viscosities(case):
    if case["shape"] == "splash":
        return 0.04, 0.6
    return 0.05, 0.5


def _batch_members(case, seed):
    """Parameters of the batch's instances; sides log-uniform, films and droplets in turn."""
    rng = np.random.default_rng(seed)
    sizes = np.random.default_rng(case["n"])  # a study's grids do not change with its data
    out = []
    for i in range(case["n"]):
        nx, ny = (int(round(math.exp(sizes.uniform(math.log(case["lo"]), math.log(case["hi"])))))
                  for _ in range(2))
        a = rng.uniform(0.125, 0.5)
        m = {"nx": nx, "ny": ny, "a": a, "T": temperature(rng.uniform(0.62, 0.88), a),
             "sigma": SIGMA * rng.uniform(0.95, 1.05), "ratio": rng.uniform(1.0, 10.0),
             "film": i % 2 == 0}
        out.append(m)
    for m, rl, rv in zip(out, *coexistences([m["a"] for m in out], [m["T"] for m in out])):
        m["rl"], m["rv"] = float(rl), float(rv)
    return out


def _member_field(m):
    y, x = torch.meshgrid(torch.arange(m["ny"], device="cuda").double(),
                          torch.arange(m["nx"], device="cuda").double(), indexing="ij")
    cx, cy = (m["nx"] - 1) / 2.0, (m["ny"] - 1) / 2.0
    if m["film"]:
        d = torch.abs(y - cy) - m["ny"] / 4.0
    else:
        d = torch.hypot(x - cx, y - cy) - min(m["nx"], m["ny"]) / 4.0
    return _profile(d, m["rl"], m["rv"]).float().cpu().numpy()


def _train_data(case, seed):
    """Rows (a, T/Tc, sigma, viscosity ratio) and five smooth targets, and initial weights."""
    rng = np.random.default_rng(seed)
    n = case["rows"]
    x = np.stack([rng.uniform(0.125, 1, n), rng.uniform(0.5, 0.9, n),
                  rng.uniform(0.09, 0.14, n), rng.uniform(1, 20, n)], axis=1)
    t = np.stack([0.01 * np.sin(5 * x[:, 1]), 0.3 * x[:, 1] - x[:, 2] * 2, 4 / np.sqrt(x[:, 0]),
                  np.log(x[:, 3]) * 0.2, np.cos(3 * x[:, 0]) + x[:, 1]], axis=1)
    t = t + 0.01 * rng.normal(size=t.shape)
    parts = []
    for fi, fo in ((4, 64), (64, 64), (64, 5)):
        k = 1.0 / math.sqrt(fi)
        parts += [rng.uniform(-k, k, fo * fi), rng.uniform(-k, k, fo)]
    return x, t, np.concatenate(parts).astype(np.float32)


def _warm_inputs(case, seed):
    rl, rv = coexistence(A_EOS, temperature(case["tr"]))
    rng = np.random.default_rng(seed)
    drops = _layout(case["nx"], case["ny"], case["drops"], rng)
    return drops, dict(rho_l=rl * (1 + 1e-4 * rng.normal()), rho_v=rv, width=4.2, shift=0.1,
                       curvature=0.4), rl, rv


# ---------------------------------------------------------------------------------------
def prepare(case, seed):
    from paper_1211_6932_gb300 import Batch, Eos, Instance, Lattice, Mlp
    from paper_1211_6932_gb300.warm import WarmParams
    stream = torch.cuda.Stream()
    if case["kind"] == "batch":
        members = _batch_members(case, seed)
        insts = [Instance(m["nx"], m["ny"], Eos(a=m["a"], T=m["T"]), sigma=m["sigma"], s=RATES,
                          nu_l=0.1, nu_v=0.1 * m["ratio"], visc_mode="linear", rho_l=m["rl"],
                          rho_v=m["rv"]) for m in members]
        return {"case": case, "batch": Batch(insts, stream=stream),
                "fields": [_member_field(m) for m in members]}
    if case["kind"] == "train":
        x, t, w = _train_data(case, seed)
        net = Mlp(w, max_rows=case["rows"], stream=stream)
        net.fit_scaling(x, t)
        net.set_data(x, t)
        return {"case": case, "net": net}
    shape = (case["ny"], case["nx"])
    T = temperature(case["tr"])
    if case["kind"] == "warm":
        drops, warm, rl, rv = _warm_inputs(case, seed)
        lat = Lattice(case["nx"], case["ny"], Eos(a=A_EOS, T=T), sigma=SIGMA, s=RATES, nu_l=0.05,
                      nu_v=0.5, visc_mode="linear", rho_l=rl, rho_v=rv, stream=stream)
        out = [torch.empty(shape, device="cuda") for _ in range(3)]
        return {"case": case, "lattice": lat, "drops": drops, "warm": WarmParams(**warm),
                "limits": (rv + 0.1 * (rl - rv), rl - 0.1 * (rl - rv)), "out": out}
    rho, ux, uy, rl, rv = _fields(case, seed)
    nu_l, nu_v = _viscosities(case) if case["visc"] != "const" else (0.0, 0.0)
    lat = Lattice(case["nx"], case["ny"], Eos(a=A_EOS, T=T), sigma=SIGMA, s=_rates(case),
                  nu_l=nu_l, nu_v=nu_v, precision=case["precision"], visc_mode=case["visc"],
                  bc=case["bc"], psi_fp64=case["psi_fp64"], rho_l=rl, rho_v=rv, stream=stream)
    state = {"case": case, "lattice": lat}
    if case["io"] == "host":
        state["fields"] = [None if f is None else f.cpu().numpy() for f in (rho, ux, uy)]
    else:
        state["fields"] = [rho, ux, uy]
        kind = torch.float64 if case["precision"] == "fp64" else torch.float32
        state["out"] = [torch.empty(shape, dtype=kind, device="cuda") for _ in range(3)]
        torch.cuda.synchronize()  # the lattice's stream reads what torch's stream wrote
    return state


def run(state):
    case = state["case"]
    if case["kind"] == "batch":
        batch = state["batch"]
        for i, rho in enumerate(state["fields"]):
            batch.init_fields(i, rho)
        batch.run_to_equilibrium(1e-12, check_every=100, max_steps=case["steps"])
        got = [batch.moments(i, dtype=np.float32) for i in range(len(batch))]
        return {k: np.concatenate([g[k].ravel() for g in got]) for k in ("rho", "ux", "uy")}
    if case["kind"] == "train":
        losses = state["net"].train(case["updates"], **ADAM)
        return {"losses": losses, "weights": state["net"].params()}
    lat = state["lattice"]
    if case["kind"] == "warm":
        lat.init_droplets(state["drops"], state["warm"], curvature=True, balanced=True)
        lat.step(case["steps"])
        vap, _, liq, _ = lat.phase_stats(*state["limits"])
        lat.moments_device(*state["out"])
        return {"rho": state["out"][0], "ux": state["out"][1], "uy": state["out"][2],
                "vapour": float(vap), "liquid": float(liq)}
    if case["io"] == "host":
        lat.init_fields(*state["fields"])
        lat.step(case["steps"])
        return lat.moments()
    lat.init_fields_device(*state["fields"])
    lat.step(case["steps"])
    lat.moments_device(*state["out"])
    return {"rho": state["out"][0], "ux": state["out"][1], "uy": state["out"][2]}


def work(case):
    """Fields in and fields out, and the arithmetic of the steps (an update has about 240
    floating-point operations, psi included).  A pass cannot do without more traffic than that
    where the state stays on the chip; a lattice larger than the caches streams its state
    besides, 72 bytes an update in FP32 when each pass over it takes one step."""
    if case["kind"] == "train":
        n = case["rows"]
        return {"bytes": 4.0 * 4805 * 3 * 2, "flops": 6.0 * 4805 * n * case["updates"]}
    if case["kind"] == "batch":
        sizes = np.random.default_rng(case["n"])
        nodes = 0
        for _ in range(case["n"]):
            nx, ny = (int(round(math.exp(sizes.uniform(math.log(case["lo"]),
                                                       math.log(case["hi"])))))
                      for _ in range(2))
            nodes += nx * ny
        return {"bytes": 16.0 * nodes, "flops": 240.0 * nodes * case["steps"]}
    nodes = case["nx"] * case["ny"]
    if case["kind"] == "warm":
        return {"bytes": 12.0 * nodes, "flops": 240.0 * nodes * (case["steps"] + 1)}
    ins = 3 if case["shape"] == "splash" else 1
    out = 8 if case["precision"] == "fp64" or case["io"] == "host" else 4
    return {"bytes": (8.0 * ins + 3.0 * out) * nodes, "flops": 240.0 * nodes * case["steps"]}


# ---------------------------------------------------------------------------------------
# The same passes in plain 64-bit torch: every lattice of a case as one flat list of nodes.
EX = (0, 1, 0, -1, 0, 1, -1, -1, 1)
EY = (0, 0, 1, 0, -1, 1, 1, -1, -1)
OPP = (0, 3, 4, 1, 2, 7, 8, 5, 6)
TW = (4 / 9,) + (1 / 9,) * 4 + (1 / 36,) * 4
MRT = torch.tensor([[1, 1, 1, 1, 1, 1, 1, 1, 1], [-4, -1, -1, -1, -1, 2, 2, 2, 2],
                    [4, -2, -2, -2, -2, 1, 1, 1, 1], [0, 1, 0, -1, 0, 1, -1, -1, 1],
                    [0, -2, 0, 2, 0, 1, -1, -1, 1], [0, 0, 1, 0, -1, 1, 1, -1, -1],
                    [0, 0, -2, 0, 2, 1, 1, -1, -1], [0, 1, -1, 1, -1, 0, 0, 0, 0],
                    [0, 0, 0, 0, 0, 1, -1, 1, -1]], dtype=torch.float64)


def _combine(coeffs, fields):
    """sum of c * f over the nonzero coefficients."""
    acc = None
    for c, f in zip(coeffs, fields):
        if c:
            acc = c * f if acc is None else acc.add_(f, alpha=c)
    return acc


class Plain:
    """Lattices (nx, ny, walls) one after another; par: tensors or numbers per node."""

    def __init__(self, sizes, par):
        self.par, at = par, 0
        nb = [[] for _ in range(9)]
        out = [[] for _ in range(9)]
        for nx, ny, walls in sizes:
            y, x = torch.meshgrid(torch.arange(ny, device="cuda"),
                                  torch.arange(nx, device="cuda"), indexing="ij")
            for q in range(1, 9):
                yy, xx = y + EY[q], (x + EX[q]) % nx
                out[q].append(((yy < 0) | (yy >= ny)).ravel() if walls else None)
                yy = yy.clamp(0, ny - 1) if walls else yy % ny
                nb[q].append((yy * nx + xx).ravel() + at)
            at += nx * ny
        self.n = at
        self.nb = [None] + [torch.cat(v) for v in nb[1:]]
        self.out = [None] + [v[0] for v in out[1:]]  # walls: single lattices only

    def start(self, rho, ux=None, uy=None):
        ux = torch.zeros_like(rho) if ux is None else ux
        uy = torch.zeros_like(rho) if uy is None else uy
        u2 = ux * ux + uy * uy
        self.f = []
        for q in range(9):
            eu = EX[q] * ux + EY[q] * uy
            self.f.append(TW[q] * rho * (1 + 3 * eu + 4.5 * eu * eu - 1.5 * u2))

    def psi(self, rho):
        p = self.par
        x = 0.25 * B_EOS * rho
        pe = rho * p["T"] * (1 + x * (1 + x * (1 - x))) / (1 - x) ** 3 - p["a"] * rho * rho
        return torch.sqrt(torch.clamp(2 * (pe - rho / 3) / G, min=0.0))

    def force(self, rho):
        psi = self.psi(rho)
        gx, gy = torch.zeros_like(psi), torch.zeros_like(psi)
        for q in range(1, 9):
            v = psi[self.nb[q]] * (1 / 3 if q <= 4 else 1 / 12)
            if EX[q]:
                gx.add_(v, alpha=EX[q])
            if EY[q]:
                gy.add_(v, alpha=EY[q])
        return psi, -G * psi * gx, -G * psi * gy

    def fields(self):
        rho = sum(self.f)
        psi, fx, fy = self.force(rho)
        jx, jy = _combine(EX, self.f), _combine(EY, self.f)
        return rho, psi, fx, fy, (jx + 0.5 * fx) / rho, (jy + 0.5 * fy) / rho

    def step(self):
        p, s = self.par, self.par["s"]
        rho, psi, fx, fy, ux, uy = self.fields()
        if p["visc"] == "const":
            s_nu = s[7]
        elif p["visc"] == "step":
            s_nu = torch.where(rho >= 0.5218 / B_EOS, 1 / (3 * p["nu_l"] + 0.5),
                               1 / (3 * p["nu_v"] + 0.5))
        else:
            fr = torch.clamp((rho - p["rho_v"]) / (p["rho_l"] - p["rho_v"]), 0.0, 1.0)
            s_nu = 1 / (3 * (p["nu_v"] + fr * (p["nu_l"] - p["nu_v"])) + 0.5)
        uf, u2 = ux * fx + uy * fy, ux * ux + uy * uy
        extra = 12 * p["sigma"] * (fx * fx + fy * fy) / torch.clamp(psi * psi, min=1e-300)
        eq = [rho, rho * (3 * u2 - 2), rho * (1 - 3 * u2), rho * ux, -rho * ux, rho * uy,
              -rho * uy, rho * (ux * ux - uy * uy), rho * ux * uy]
        src = [None, 6 * uf + extra / (1 / s[1] - 0.5), -6 * uf - extra / (1 / s[2] - 0.5), fx,
               -fx, fy, -fy, 2 * (ux * fx - uy * fy), ux * fy + uy * fx]
        delta = []
        for k in range(9):
            sk = s_nu if k >= 7 else s[k]
            m = _combine(MRT[k].tolist(), self.f)
            d = (eq[k] - m) * sk
            if src[k] is not None:
                d = d + (1 - 0.5 * sk) * src[k]
            delta.append(d / float((MRT[k] ** 2).sum()))
        post = []
        for q in range(9):
            post.append(self.f[q] + _combine(MRT[:, q].tolist(), delta))
        for q in range(9):
            if q == 0:
                self.f[0] = post[0]
                continue
            o = OPP[q]
            v = post[q][self.nb[o]]
            self.f[q] = v if self.out[o] is None else torch.where(self.out[o], post[o], v)

    def answer(self):
        rho, _, _, _, ux, uy = self.fields()
        return {"rho": rho, "ux": ux, "uy": uy}


def exact(case, seed):
    if case["kind"] == "train":
        return _exact_train(case, seed)
    if case["kind"] == "batch":
        members = _batch_members(case, seed)
        n = [m["nx"] * m["ny"] for m in members]

        def per_node(values):
            return torch.repeat_interleave(torch.tensor(values, dtype=torch.float64, device="cuda"),
                                           torch.tensor(n, device="cuda"))
        par = {"a": per_node([m["a"] for m in members]), "T": per_node([m["T"] for m in members]),
               "sigma": per_node([m["sigma"] for m in members]), "s": RATES, "visc": "linear",
               "nu_l": 0.1, "nu_v": per_node([0.1 * m["ratio"] for m in members]),
               "rho_l": per_node([m["rl"] for m in members]),
               "rho_v": per_node([m["rv"] for m in members])}
        ref = Plain([(m["nx"], m["ny"], False) for m in members], par)
        ref.start(torch.cat([torch.from_numpy(_member_field(m)).double().cuda().ravel()
                             for m in members]))
        for _ in range(case["steps"]):
            ref.step()
        return ref.answer()
    nx, ny = case["nx"], case["ny"]
    T = temperature(case["tr"])
    par = {"a": A_EOS, "T": T, "sigma": SIGMA}
    if case["kind"] == "warm":
        drops, warm, rl, rv = _warm_inputs(case, seed)
        par |= {"s": RATES, "visc": "linear", "nu_l": 0.05, "nu_v": 0.5, "rho_l": rl, "rho_v": rv}
        kappa = float(np.mean(1.0 / drops[:, 2]))
        ro = warm["rho_v"] * (1 + warm["curvature"] * kappa)
        h = 1e-5
        slope = (_p(warm["rho_l"] + h, A_EOS, T) - _p(warm["rho_l"] - h, A_EOS, T)) / (2 * h)
        ri = warm["rho_l"] + (_p(ro, A_EOS, T) - _p(warm["rho_v"], A_EOS, T)) / slope
        rho = _drops_field(nx, ny, drops, ri, ro, warm["shift"], warm["width"]).ravel()
        ref = Plain([(nx, ny, False)], par)
        _, fx, fy = ref.force(rho)
        ref.start(rho, -0.5 * fx / rho, -0.5 * fy / rho)
        for _ in range(case["steps"]):
            ref.step()
        got = {k: v.view(ny, nx) for k, v in ref.answer().items()}
        lo, hi = rv + 0.1 * (rl - rv), rl - 0.1 * (rl - rv)
        got["vapour"] = float(got["rho"][got["rho"] < lo].mean())
        got["liquid"] = float(got["rho"][got["rho"] > hi].mean())
        return got
    rho, ux, uy, rl, rv = _fields(case, seed)
    nu_l, nu_v = _viscosities(case)
    par |= {"s": _rates(case), "visc": case["visc"], "nu_l": nu_l, "nu_v": nu_v, "rho_l": rl,
            "rho_v": rv}
    ref = Plain([(nx, ny, case["bc"] == "walls")], par)
    ref.start(rho.ravel(), None if ux is None else ux.ravel(), None if uy is None else uy.ravel())
    for _ in range(case["steps"]):
        ref.step()
    return {k: v.view(ny, nx) for k, v in ref.answer().items()}


def _exact_train(case, seed):
    """Full-batch Adam on the mean squared error of the standardised outputs, the forward and
    backward passes at weights rounded to bfloat16."""
    x, t, w = _train_data(case, seed)
    x, t = torch.from_numpy(x), torch.from_numpy(t)
    xn = (x - x.mean(0)) / x.std(0, unbiased=False)
    tn = (t - t.mean(0)) / t.std(0, unbiased=False)
    p = torch.from_numpy(w).double()
    m, v = torch.zeros_like(p), torch.zeros_like(p)
    sizes = (256, 64, 4096, 64, 320, 5)
    losses = []
    for k in range(1, case["updates"] + 1):
        q = p.float().bfloat16().double().requires_grad_(True)
        w1, b1, w2, b2, w3, b3 = torch.split(q, sizes)
        h = torch.nn.functional.gelu(xn @ w1.view(64, 4).T + b1)
        h = torch.nn.functional.gelu(h @ w2.view(64, 64).T + b2)
        loss = ((h @ w3.view(5, 64).T + b3 - tn) ** 2).mean()
        g, = torch.autograd.grad(loss, q)
        losses.append(float(loss.detach()))
        m = ADAM["beta1"] * m + (1 - ADAM["beta1"]) * g
        v = ADAM["beta2"] * v + (1 - ADAM["beta2"]) * g * g
        p = p - ADAM["lr"] * (m / (1 - ADAM["beta1"] ** k)) / (
            torch.sqrt(v / (1 - ADAM["beta2"] ** k)) + ADAM["eps"])
    return {"losses": np.array(losses), "weights": p.numpy()}
