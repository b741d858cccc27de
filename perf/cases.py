"""The work that users of the library have it do, as cases that can be timed and checked.

A case advances lattices (or runs one of the passes around them) through the package's public
entry points. `listed()` holds the fixed cases, `draw()` gives more of the same ranges,
`prepare()` builds what a user's program holds before the call, `run()` is one pass, `work()` its
unavoidable bytes and operations, `exact()` the outputs in 64-bit arithmetic, written here from
the scheme's equations in plain torch.

Kinds of case:
  steps   one lattice: lb_step(n), then its moment fields (and, with `monitor`, the mass / residual
          reduction a run to the steady state polls)
  batch   a sweep of independent 8-wide channels advanced by one launch, then every channel's
          density and velocity
  stream  the D2Q9 stream-and-collide scheme on a periodic box, then its moment fields
  host    host-resident state: upload the compact state, one step, read the state back
  place   learned placement on a lattice: features of every node, then the network's p
  train   mini-batch training of the placement network, one epoch
"""
from __future__ import annotations

import math

import numpy as np
import torch

SQRT3 = math.sqrt(3.0)
TILE = 128          # region maps are quantised to tiles of 128 columns x 1 row (include/lb.h)
ON_CHIP = 32 << 20  # a state up to this size can stay in the chip's shared memory between steps
FIELDS = 9          # moment fields of lb_moments
NPARAM = 4801       # parameters of the placement network


# --------------------------------------------------------------------------- cases

def listed():
    return [
        # the smallest run: plane Couette flow, 4 columns, FP64 (the accuracy studies)
        dict(name="couette_4x32_f64", kind="steps", flow="couette", nx=4, ny=32, rows=4, kn=0.1, store="f64", steps=50),
        # a steady channel of the learned-placement study, polled for convergence
        dict(name="channel_8x64_monitored", kind="steps", flow="force", nx=8, ny=64, rows=10, kn=0.03,
             store="f32_dev", steps=100, monitor=True),
        # ragged width, the package's default storage
        dict(name="channel_300x37_f32", kind="steps", flow="force", nx=300, ny=37, rows=5, kn=0.1, store="f32", steps=20),
        # the force-driven Poiseuille channel
        dict(name="poiseuille_1024x512", kind="steps", flow="force", nx=1024, ny=512, rows=32, kn=0.1, store="f32_dev",
             steps=20),
        # the pressure-driven long channel: the headline workload, and its 16-bit form
        dict(name="long_16384x128", kind="steps", flow="long", nx=16384, ny=128, kn=0.2, store="f32_dev", steps=20),
        dict(name="long_16384x128_f16", kind="steps", flow="long", nx=16384, ny=128, kn=0.2, store="f16_dev", steps=20),
        # the most accurate 16-bit form: stochastic rounding, per-column reference density
        dict(name="long_4096x128_bf16_sr", kind="steps", flow="long", nx=4096, ny=128, kn=0.2, store="bf16_dev",
             rounding="stochastic", col=True, steps=20),
        # the sweep of 512 channels of uneven height and Kn
        dict(name="batch_512", kind="batch", n=512, ny_lo=16, ny_hi=256, store="f32_dev", steps=500),
        # stream-and-collide on a periodic box
        dict(name="stream_2048x1024", kind="stream", nx=2048, ny=1024, kn=0.02, store="f32_dev", steps=20),
        # state resident on the host: upload, step, read back
        dict(name="host_16384x128", kind="host", nx=16384, ny=128, kn=0.2, store="f32_dev"),
        # one evaluation of the placement network over the long channel
        dict(name="place_16384x128", kind="place", nx=16384, ny=128, kn=0.2, store="f32_dev"),
        # one epoch on the sample count of the placement study
        dict(name="train_100000", kind="train", n=100000, batch=256),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["small", "small", "wide", "wide", "long", "long", "batch", "stream", "host", "place", "train"])
    if kind == "small":     # the channels of accuracy and placement studies
        store = rng.choice(["f64", "f32", "f32_dev", "f32_dev", "f16_dev", "bf16_dev"])
        ny = _log_int(rng, 16, 300)
        return dict(kind="steps", flow=rng.choice(["couette", "force", "oscillating", "kramers"]), nx=_log_int(rng, 4, 128),
                    ny=ny, rows=max(2, int(round(rng.uniform(0.08, 0.2) * ny))), kn=10.0 ** rng.uniform(-1.5, -0.3),
                    store=store, sets=rng.choice([36, 36, 16]), steps=rng.randint(20, 120), monitor=rng.random() < 0.3)
    if kind == "wide":      # two-dimensional channels, any width
        store = rng.choice(["f32", "f32_dev", "f32_dev", "f16_dev", "bf16_dev"])
        ny = _log_int(rng, 24, 512)
        return dict(kind="steps", flow=rng.choice(["couette", "force"]), nx=_log_int(rng, 140, 2048), ny=ny,
                    rows=max(2, int(round(rng.uniform(0.04, 0.15) * ny))), kn=10.0 ** rng.uniform(-1.5, -0.3), store=store,
                    sets=rng.choice([36, 36, 16]), steps=rng.randint(5, 20))
    if kind == "long":      # pressure-driven channels
        store = rng.choice(["f32_dev", "f32_dev", "f16_dev", "bf16_dev"])
        sr = store != "f32_dev" and rng.random() < 0.5
        return dict(kind="steps", flow="long", nx=_log_int(rng, 256, 16384), ny=_log_int(rng, 32, 128),
                    kn=rng.uniform(0.05, 0.4), store=store, rounding="stochastic" if sr else "nearest",
                    col=rng.random() < 0.3, steps=rng.randint(5, 20))
    if kind == "batch":
        hi = rng.randint(64, 256)
        return dict(kind="batch", n=_log_int(rng, 16, 512), ny_lo=16, ny_hi=hi,
                    store=rng.choice(["f32_dev", "f32_dev", "f32", "bf16_dev"]), steps=rng.randint(50, 300))
    if kind == "stream":
        return dict(kind="stream", nx=_log_int(rng, 64, 2048), ny=_log_int(rng, 16, 1024), kn=10.0 ** rng.uniform(-1.7, -0.5),
                    store=rng.choice(["f32_dev", "f32_dev", "f32", "f16_dev"]), steps=rng.randint(5, 20))
    if kind == "host":
        return dict(kind="host", nx=_log_int(rng, 300, 16384), ny=_log_int(rng, 32, 128), kn=rng.uniform(0.05, 0.4),
                    store=rng.choice(["f32_dev", "f32_dev", "f16_dev"]))
    if kind == "place":
        return dict(kind="place", nx=_log_int(rng, 300, 16384), ny=_log_int(rng, 32, 128), kn=rng.uniform(0.05, 0.4),
                    store=rng.choice(["f32_dev", "f32"]))
    return dict(kind="train", n=_log_int(rng, 2000, 100000), batch=rng.choice([64, 128, 200, 256, 500, 512]))


# --------------------------------------------------------------------------- inputs

class _Flow:
    """Geometry, parameters and start of one lattice (the fields lb_create wants)."""

    def __init__(self, **kw):
        self.sets, self.tau_mode, self.iface, self.rho0, self.cfl, self.gx, self.gy = (9, 36), 0, "hermite", 1.0, 0.5, 0.0, 0.0
        self.rho_ref = 1.0
        self.__dict__.update(kw)


def _bands(nx, ny, bottom, top):
    m = np.zeros((ny, nx), np.uint8)
    m[:bottom] = 1
    if top:
        m[ny - top:] = 1
    return m


def _waves(rng, nx, ny, n=3):
    """A smooth field of unit size: a few low modes (periodic in x, zero at the walls)."""
    x, y = 2 * np.pi * np.arange(nx) / nx, np.pi * np.arange(ny) / max(ny - 1, 1)
    out = np.zeros((ny, nx))
    for _ in range(n):
        k, m, ph = int(rng.integers(1, 4)), int(rng.integers(1, 5)), rng.uniform(0, 2 * np.pi)
        out += np.outer(np.sin(m * y), np.sin(k * x + ph)) / n
    return out


def _flow(case, seed):
    """The channel of a steps / host / place case with its seeded start."""
    rng = np.random.default_rng(seed)
    nx, ny, kn = case["nx"], case["ny"], case["kn"]
    flow = case.get("flow", "long")
    sets = (9, case.get("sets", 36))
    rho, ux, uy = np.ones((ny, nx)), np.zeros((ny, nx)), np.zeros((ny, nx))
    y = np.arange(ny) / (ny - 1)
    if flow == "long":
        # pressure-driven: density ratio 2, the local-Kn region map, the lubrication estimate
        x = np.arange(nx) / (nx - 1)
        est = np.sqrt(4.0 - 3.0 * x)
        kn_x = kn / est
        d = np.minimum(np.arange(ny), ny - 1 - np.arange(ny)) / (ny - 1)
        m = (kn_x[None, :] / np.maximum(d[:, None], 1e-300) > 0.2 / 0.15).astype(np.uint8)
        m[:2], m[ny - 2:] = 1, 1
        rho = np.broadcast_to(est, (ny, nx)).copy()
        ux = (-np.gradient(est, 1.0 / (ny - 1))[None, :] / (2.0 * kn)) * ((y * (1 - y))[:, None] + 2.8 * kn_x[None, :])
        f = _Flow(region_map=m, kn_ref=kn, rho0=1.5, walls={
            "bottom": {"kind": "diffuse"}, "top": {"kind": "diffuse"},
            "left": {"kind": "pressure", "rho": 2.0}, "right": {"kind": "pressure", "rho": 1.0}})
        f.col = est
    else:
        rows = case["rows"]
        uw = SQRT3 * rng.uniform(0.02, 0.06)
        f = _Flow(region_map=_bands(nx, ny, rows, 0 if flow == "kramers" else rows), kn_ref=kn)
        b, t = {"kind": "diffuse"}, {"kind": "diffuse"}
        if flow == "couette":
            b["ux"], t["ux"] = -uw, uw
        elif flow == "oscillating":
            b["ux"], b["omega"] = uw, 1.0
        elif flow == "kramers":
            t["ux"] = uw
            ux += (uw * y)[:, None]
        else:
            f.gx = 8.0 * kn * uw
        f.walls = {"bottom": b, "top": t}
    # 0.38 keeps high-order bands of any thickness stable under two-dimensional disturbances; the
    # thin bands of the long channel run at 0.5
    f.nx, f.ny, f.sets, f.cfl = nx, ny, sets, 0.5 if flow == "long" and case["kind"] != "place" else 0.38
    f.init = (rho * (1.0 + 0.01 * _waves(rng, nx, ny)), ux + 0.02 * _waves(rng, nx, ny), uy + 0.01 * _waves(rng, nx, ny))
    return f


def _sweep(case, seed):
    """Independent Couette / force-driven channels of uneven height and Kn."""
    rng = np.random.default_rng(seed)
    # heights are drawn once per case, so that every seed has the same amount of work
    hs = np.random.default_rng(1007).integers(case["ny_lo"], case["ny_hi"] + 1, case["n"])
    out = []
    for ny in hs:
        ny = int(ny)
        kn, u = float(10.0 ** rng.uniform(-1.9, 0.0)), SQRT3 * float(rng.uniform(0.01, 0.1))
        rows = max(2, int(round(0.15 * ny)))
        couette = rng.random() < 0.5
        walls = {"bottom": {"kind": "diffuse"}, "top": {"kind": "diffuse"}}
        if couette:
            walls["bottom"]["ux"], walls["top"]["ux"] = -u, u
        out.append(_Flow(nx=8, ny=ny, cfl=0.38, region_map=_bands(8, ny, rows, rows), kn_ref=kn, gx=0.0 if couette else 8.0 * kn * u,
                         walls=walls, init=(1.0 + 0.01 * _waves(rng, 8, ny), 0.02 * _waves(rng, 8, ny),
                                            0.01 * _waves(rng, 8, ny))))
    return out


def _box(case, seed):
    """A periodic box with a few waves of velocity and density."""
    rng = np.random.default_rng(seed)
    nx, ny = case["nx"], case["ny"]
    x, y = 2 * np.pi * np.arange(nx) / nx, 2 * np.pi * np.arange(ny) / ny

    def waves():
        out = np.zeros((ny, nx))
        for _ in range(3):
            k, m, ph, ps = int(rng.integers(1, 4)), int(rng.integers(1, 4)), rng.uniform(0, 6.28), rng.uniform(0, 6.28)
            out += np.outer(np.sin(m * y + ps), np.sin(k * x + ph)) / 3
        return out
    side = {"kind": "periodic"}
    return _Flow(nx=nx, ny=ny, region_map=np.zeros((ny, nx), np.uint8), kn_ref=case["kn"], sets=(9, 36),
                 walls={"bottom": side, "top": side, "left": side, "right": side},
                 init=(1.0 + 0.02 * waves(), 0.1 * waves(), 0.1 * waves()))


def _samples(case, seed):
    """Node samples x [8][n] of the size and spread of the placement features, labels y [n] from
    a smooth rule with a few flipped, and the network's start."""
    g = torch.Generator(device="cuda").manual_seed(int(seed))
    n = case["n"]
    z = torch.randn(8, n, generator=g, device="cuda")
    y = ((z[0] * z[1] + 0.5 * z[2].abs() + 0.3 * z[6] + 0.1 * torch.randn(n, generator=g, device="cuda")) > 0.4).float()
    mean = torch.tensor([0.0, 0.01, 0.0, 0.001, 0.0, 0.25, 0.15, 0.002], device="cuda")
    scale = torch.tensor([0.004, 0.02, 0.004, 0.002, 0.001, 0.15, 0.04, 0.001], device="cuda")
    x = (z * scale[:, None] + mean[:, None]).contiguous()
    rng = np.random.default_rng(seed)
    params = np.concatenate([rng.standard_normal(512) * 0.5, np.zeros(64), rng.standard_normal(4096) * math.sqrt(2 / 64),
                             np.zeros(64), rng.standard_normal(64) * math.sqrt(2 / 64), np.zeros(1)]).astype(np.float32)
    return x, y, params, torch.cat([mean, scale]).cpu().numpy().astype(np.float32)


def _network(seed):
    """Weights of a placement network and the feature means and scales it was trained with."""
    rng = np.random.default_rng(seed + 77)
    params = np.concatenate([rng.standard_normal(512) * 0.5, rng.standard_normal(64) * 0.1,
                             rng.standard_normal(4096) * math.sqrt(2 / 64), rng.standard_normal(64) * 0.1,
                             rng.standard_normal(64) * math.sqrt(2 / 64), np.zeros(1)]).astype(np.float32)
    norm = np.array([0.0, 0.0, 0.0, 0.0, 0.0, 0.25, 0.15, 0.003, 0.01, 0.05, 0.01, 0.01, 0.01, 0.15, 0.04, 0.005], np.float32)
    return params, norm


# --------------------------------------------------------------------------- the library

def _lattice(f, case, **kw):
    import paper_1007_4895_gb300 as lb
    if case.get("col"):
        kw["rho0_col"] = f.col
    lat = lb.Lattice(f.nx, f.ny, f.region_map, sets=f.sets, kn_ref=f.kn_ref, rho_ref=f.rho_ref, walls=f.walls,
                     store=case["store"], iface=f.iface, rho0=f.rho0, gx=f.gx, gy=f.gy, cfl=f.cfl,
                     rounding=case.get("rounding", "nearest"), **kw)
    lat.init_equilibrium(*f.init)
    return lat


def _fields(case, nx, ny, k=FIELDS):
    return torch.empty((k, ny, nx), dtype=torch.float64 if case["store"] == "f64" else torch.float32, device="cuda")


PLACE_STEPS, HOST_STEPS = 10, 4   # steps run before a place / host pass


def prepare(case, seed):
    import paper_1007_4895_gb300 as lb
    kind = case["kind"]
    if kind == "train":
        x, y, params, norm = _samples(case, seed)
        return dict(case=case, net=lb.MLP(params, norm), x=x, y=y)
    if kind == "batch":
        fs = _sweep(case, seed)
        b = lb.Batch(fs, store=case["store"])
        return dict(case=case, batch=b, out=[_fields(case, f.nx, f.ny, 3) for f in fs])
    if kind == "stream":
        f = _box(case, seed)
        lat = _lattice(f, case, scheme="stream")
        return dict(case=case, lat=lat, out=_fields(case, f.nx, f.ny))
    f = _flow(case, seed)
    lat = _lattice(f, case)
    if kind == "steps":
        return dict(case=case, lat=lat, out=_fields(case, f.nx, f.ny))
    if kind == "place":
        lat.step(PLACE_STEPS)
        params, norm = _network(seed)
        return dict(case=case, lat=lat, net=lb.MLP(params, norm),
                    feat=torch.empty((8, f.ny, f.nx), dtype=torch.float32, device="cuda"),
                    p=torch.empty(f.ny * f.nx, dtype=torch.float32, device="cuda"))
    lat.step(HOST_STEPS)
    nb = lat.state_bytes()
    dt = torch.float16 if case["store"] == "f16_dev" else torch.float32
    src, dst = (torch.empty(nb // dt.itemsize, dtype=dt, pin_memory=True) for _ in range(2))
    lb.lb_state_store(lat.ctx, src.data_ptr(), nb)
    return dict(case=case, lat=lat, src=src, dst=dst, nbytes=nb)


def run(state):
    import paper_1007_4895_gb300 as lb
    case = state["case"]
    kind = case["kind"]
    if kind in ("steps", "stream"):
        lat = state["lat"]
        lat.step(case["steps"])
        lat.moments_into(state["out"])
        if case.get("monitor"):
            r = lat.reductions()
            return dict(fields=state["out"], mass=float(r["mass"]), residual=float(r["residual"]),
                        nonfinite=int(r["nonfinite"]), step=int(r["step"]))
        return state["out"]
    if kind == "batch":
        b = state["batch"]
        b.step(case["steps"])
        for i, t in enumerate(state["out"]):
            b.lattice(i).moments_into(t, mask=0b111)
        return torch.cat([t.flatten(1) for t in state["out"]], dim=1)
    if kind == "host":
        lat, n = state["lat"], state["nbytes"]
        lb.lb_state_load(lat.ctx, state["src"].data_ptr(), n)
        lat.step(1)
        lb.lb_state_store(lat.ctx, state["dst"].data_ptr(), n)
        return state["dst"]
    if kind == "place":
        state["lat"].features_into(state["feat"])
        state["net"].infer(state["feat"], state["p"])
        return dict(features=state["feat"], p=state["p"])
    loss = state["net"].train(state["x"], state["y"], epochs=1, batch=case["batch"], lr=1e-3, seed=1007)
    return dict(params=state["net"].params(), loss=float(loss))


# --------------------------------------------------------------------------- work

def _populations(fs):
    """Population values of the lattices `fs`, every node in its own set (tile-quantised map)."""
    n = 0
    for f in fs:
        high = int(_tiles(f.region_map).sum())
        n += f.sets[1] * high + f.sets[0] * (f.nx * f.ny - high)
    return n


def work(case):
    """Bytes: the state read and written once per call, or once per step where it is larger than
    the chip can hold between steps; inputs and outputs once. Operations of the update: 45 per
    population (moments 3, equilibrium and force 8, four limited fluxes 28, update 6), of the
    stream-and-collide update 17."""
    kind = case["kind"]
    size = {"f64": 8, "f32": 4, "f32_dev": 4}.get(case.get("store"), 2)
    if kind == "train":
        return dict(bytes=case["n"] * 36.0 + 4.0 * NPARAM * 6, flops=case["n"] * 6.0 * NPARAM)
    if kind == "place":
        nodes = case["nx"] * case["ny"]
        pops = _populations([_flow(case, 0)])
        return dict(bytes=size * pops + nodes * (8 * 4 + 4.0), flops=nodes * (2.0 * NPARAM) + 20.0 * pops)
    if kind == "stream":
        nodes = case["nx"] * case["ny"]
        state = 9 * nodes * size
        trips = case["steps"] if state > ON_CHIP else 1
        return dict(bytes=2.0 * state * trips + nodes * FIELDS * 4.0, flops=17.0 * 9 * nodes * case["steps"])
    fs = _sweep(case, 0) if kind == "batch" else [_flow(case, 0)]
    pops, nodes = _populations(fs), sum(f.nx * f.ny for f in fs)
    state = pops * size
    if kind == "host":
        return dict(bytes=4.0 * state, flops=45.0 * pops)
    # each channel of a sweep is small enough to stay on the chip for all its steps
    trips = case["steps"] if state > ON_CHIP and kind != "batch" else 1
    fields = 3 if kind == "batch" else FIELDS
    return dict(bytes=2.0 * state * trips + nodes * fields * (8.0 if size == 8 else 4.0), flops=45.0 * pops * case["steps"])


# --------------------------------------------------------------------------- 64-bit reference

def _tiles(m):
    """The region map as run: a 128-column tile of a row is high-order if any node asks for it."""
    ny, nx = m.shape
    nt = -(-nx // TILE)
    pad = np.zeros((ny, nt * TILE), bool)
    pad[:, :nx] = m > 0
    return np.repeat(pad.reshape(ny, nt, TILE).any(-1), TILE, axis=1)[:, :nx]


def _set(q):
    """Product Gauss-Hermite set, population iy * n + ix, abscissae ascending."""
    n = int(round(math.sqrt(q)))
    r, w = np.polynomial.hermite_e.hermegauss(n)
    w = w / w.sum()
    return n, np.tile(r, n), np.repeat(r, n), np.outer(w, w).ravel()


class _Exact:
    """The multiscale scheme in 64 bits for lattices of one width, stacked along y: Hermite
    equilibrium and force, tau = Kn rho_ref / rho, forward Euler with TVD minmod fluxes, diffuse
    walls, pressure columns, second-order Hermite views across the interface of the two sets."""

    def __init__(self, fs, dev):
        self.dev = dev
        T = lambda a: torch.tensor(np.asarray(a, dtype=np.float64), device=dev)  # noqa: E731
        self.q, f0 = fs[0].sets, fs[0]
        self.nx = f0.nx
        self.sets = []
        for q in self.q:
            n, cx, cy, w = _set(q)
            self.sets.append((n, T(cx)[:, None, None], T(cy)[:, None, None], T(w)[:, None, None]))
        self.xmax = max(float(s[1].abs().max()) for s in self.sets)
        self.cfl = f0.cfl
        self.map = torch.tensor(np.concatenate([_tiles(f.region_map) for f in fs]), device=dev)
        rows, self.walls, j0 = {d: [] for d in (-2, -1, 1, 2)}, [[], []], 0
        h, kn, gx = [], [], []
        for f in fs:
            for d in rows:
                rows[d].append(j0 + np.clip(np.arange(f.ny) + d, 0, f.ny - 1))
            for k, side in enumerate(("bottom", "top")):
                wl = f.walls[side]
                self.walls[k].append((j0 if k == 0 else j0 + f.ny - 1, wl.get("ux", 0.0), wl.get("omega", 0.0)))
            h += [1.0 / (f.ny - 1)] * f.ny
            kn += [f.kn_ref] * f.ny
            gx += [f.gx] * f.ny
            j0 += f.ny
        self.rows = {d: torch.tensor(np.concatenate(r), device=dev) for d, r in rows.items()}
        self.dt, self.kn, self.gx = (T(v)[:, None] for v in (np.array(h) * self.cfl / self.xmax, kn, gx))
        self.side = [f0.walls.get(s, {}).get("rho") if f0.walls.get(s, {}).get("kind") == "pressure" else None
                     for s in ("left", "right")]
        self.periodic = self.side[0] is None
        self.step_count = 0
        init = [T(np.concatenate([np.broadcast_to(f.init[k], (f.ny, f.nx)) for f in fs])) for k in range(3)]
        self.f = [self.feq(s, *init) for s in (0, 1)]
        self.pressure()

    def feq(self, s, rho, ux, uy):
        _, cx, cy, w = self.sets[s]
        e = cx * ux + cy * uy
        return w * rho * (1.0 + e + 0.5 * (e * e - (ux * ux + uy * uy)))

    def sums(self, f):
        """rho, u of every node from its own set."""
        out = []
        for s in (0, 1):
            _, cx, cy, _ = self.sets[s]
            r = f[s].sum(0)
            out.append((r, (f[s] * cx).sum(0) / r, (f[s] * cy).sum(0) / r))
        return tuple(torch.where(self.map, b, a) for a, b in zip(*out))

    def project(self, f, s):
        """Values of set 1 - s as their second-order Hermite expansion in set s."""
        _, ox, oy, _ = self.sets[1 - s]
        _, cx, cy, w = self.sets[s]
        a0, ax, ay = f.sum(0), (f * ox).sum(0), (f * oy).sum(0)
        xx, xy, yy = (f * (ox * ox - 1)).sum(0), (f * (ox * oy)).sum(0), (f * (oy * oy - 1)).sum(0)
        return w * (a0 + ax * cx + ay * cy + 0.5 * (xx * (cx * cx - 1) + 2 * xy * cx * cy + yy * (cy * cy - 1)))

    def views(self):
        for s in (0, 1):
            own = self.map if s else ~self.map
            yield s, torch.where(own, self.f[s], self.project(self.f[1 - s], s))

    def pressure(self):
        for side, (b, i) in enumerate(((0, 1), (self.nx - 1, self.nx - 2))):
            if self.side[side] is None:
                continue
            rest = slice(1, self.map.shape[0] - 1)
            own_i = self.map[:, i]
            for s in (0, 1):
                f = self.f[s][:, :, i:i + 1]
                g = self.project(self.f[1 - s][:, :, i:i + 1], s)
                f = torch.where((own_i if s else ~own_i)[:, None], f, g)
                _, cx, cy, _ = self.sets[s]
                r = f.sum(0)
                ux, uy = (f * cx).sum(0) / r, (f * cy).sum(0) / r
                v = self.feq(s, torch.full_like(r, self.side[side]), ux, uy) + f - self.feq(s, r, ux, uy)
                self.f[s][:, rest, b:b + 1] = v[:, rest]

    def shift_x(self, f, k):
        """f at column i + k."""
        if self.periodic:
            return torch.roll(f, -k, -1)
        i = (torch.arange(self.nx, device=self.dev) + k).clamp(0, self.nx - 1)
        return f.index_select(-1, i)

    @staticmethod
    def limited(a, b, c, d, k):
        """Difference of the two limited face values along the window a, b, c (node), d, upwind first."""
        mm = lambda p, q: torch.where(p * q > 0, torch.where(p.abs() < q.abs(), p, q), torch.zeros_like(p))  # noqa: E731
        d0, d1, d2 = b - a, c - b, d - c
        return d1 + k * (mm(d1, d2) - mm(d0, d1))

    def step(self, n):
        for _ in range(n):
            rho, ux, uy = self.sums(self.f)
            om = self.dt * rho / self.kn
            new = []
            for s, v in self.views():
                m, cx, cy, w = self.sets[s]
                e = cx * ux + cy * uy
                g = om * (self.feq(s, rho, ux, uy) - v) + self.dt * w * rho * self.gx * (cx + cx * e - ux) + v
                v4, g4 = v.view(m, m, *v.shape[1:]), g.view(m, m, *v.shape[1:])
                r = cx[:m, 0, 0].tolist()
                for i, x in enumerate(r):
                    c, d = abs(x) * self.cfl / self.xmax, 1 if x > 0 else -1
                    if c < 1e-12:
                        continue
                    p = v4[:, i]
                    g4[:, i] -= c * self.limited(self.shift_x(p, -2 * d), self.shift_x(p, -d), p, self.shift_x(p, d), 0.5 * (1 - c))
                    p = v4[i]
                    g4[i] -= c * self.limited(p.index_select(1, self.rows[-2 * d]), p.index_select(1, self.rows[-d]), p,
                                              p.index_select(1, self.rows[d]), 0.5 * (1 - c))
                new.append(g)
            self.f, self.step_count = new, self.step_count + 1
            for k, walls in enumerate(self.walls):
                j = torch.tensor([wl[0] for wl in walls], device=self.dev)
                t = (self.step_count * self.dt[j, 0]).tolist()
                uw = torch.tensor([u * (math.sin(o * tt) if o > 0 else 1.0) for (_, u, o), tt in zip(walls, t)],
                                  dtype=torch.float64, device=self.dev)[:, None].expand(-1, self.nx)
                for s in (0, 1):
                    xn = self.sets[s][2] * (1.0 if k == 0 else -1.0)
                    f = self.f[s][:, j]
                    wall = self.feq(s, torch.ones_like(uw), uw, torch.zeros_like(uw))
                    rho_w = (f * (-xn).clamp(min=0)).sum(0) / (wall * xn.clamp(min=0)).sum(0)
                    self.f[s][:, j] = torch.where(xn > 0, rho_w * wall, f)
            self.pressure()
        return self

    def fields(self):
        rho, ux, uy = self.sums(self.f)
        both = []
        for s in (0, 1):
            _, cx, cy, _ = self.sets[s]
            f = self.f[s]
            ne = f - self.feq(s, rho, ux, uy)
            dx, dy = cx - ux, cy - uy
            d2 = dx * dx + dy * dy
            both.append(torch.stack([rho, ux, uy, (f * dx * dy).sum(0), (ne * cx * cx).sum(0), (ne * cx * cy).sum(0),
                                     (ne * cy * cy).sum(0), 0.5 * (f * d2 * dx).sum(0), 0.5 * (f * d2 * dy).sum(0)]))
        return torch.where(self.map, both[1], both[0])


def _exact_box(f, case, dev):
    """Stream-and-collide of the D2Q9 set in 64 bits: fields after the steps."""
    _, cx, cy, w = _set(9)
    T = lambda a: torch.tensor(np.asarray(a, dtype=np.float64), device=dev)  # noqa: E731
    cx, cy, w = (T(a)[:, None, None] for a in (cx, cy, w))
    h = 1.0 / f.ny
    dt = h / SQRT3

    def feq(rho, ux, uy):
        e = cx * ux + cy * uy
        return w * rho * (1.0 + e + 0.5 * (e * e - (ux * ux + uy * uy)))

    def sums(g):
        r = g.sum(0)
        return r, (g * cx).sum(0) / r, (g * cy).sum(0) / r
    g = feq(*(T(a) for a in f.init))
    for _ in range(case["steps"]):
        g = torch.stack([torch.roll(g[a], (a // 3 - 1, a % 3 - 1), (0, 1)) for a in range(9)])
        rho, ux, uy = sums(g)
        g = g + (dt * rho / f.kn_ref) * (feq(rho, ux, uy) - g)
    rho, ux, uy = sums(g)
    ne, dx, dy = g - feq(rho, ux, uy), cx - ux, cy - uy
    d2 = dx * dx + dy * dy
    return torch.stack([rho, ux, uy, (g * dx * dy).sum(0), (ne * cx * cx).sum(0), (ne * cx * cy).sum(0),
                        (ne * cy * cy).sum(0), 0.5 * (g * d2 * dx).sum(0), 0.5 * (g * d2 * dy).sum(0)])


def _exact_features(f, m):
    """The placement features from moment fields: stress and heat flux per mass, wall distance,
    local Kn, Kn |grad rho| / rho."""
    rho = m[0]
    ny, nx = rho.shape
    h = 1.0 / (ny - 1)
    gy, gx = torch.gradient(rho, spacing=h)
    j = torch.arange(ny, dtype=torch.float64, device=rho.device)
    kn = f.kn_ref / rho
    dist = torch.minimum(j, ny - 1 - j)[:, None].expand(ny, nx) * h
    return torch.stack([m[4] / rho, m[5] / rho, m[6] / rho, m[7] / rho, m[8] / rho, dist, kn,
                        kn * (gx * gx + gy * gy).sqrt() / rho])


def _unpack(th):
    return (th[:512].view(64, 8), th[512:576], th[576:4672].view(64, 64), th[4672:4736], th[4736:4800], th[4800])


def _logit(th, x):
    """The network on normalised features x [n][8]: 8 -> 64 -> 64 -> 1 with GELU."""
    w1, b1, w2, b2, w3, b3 = _unpack(th)
    g = torch.nn.functional.gelu
    return g(g(x @ w1.T + b1) @ w2.T + b2) @ w3 + b3


class _MT64:
    """The 64-bit Mersenne twister (Matsumoto & Nishimura 2000), the generator of the shuffle."""

    def __init__(self, seed):
        s = [seed & (2 ** 64 - 1)]
        for i in range(1, 312):
            s.append((6364136223846793005 * (s[-1] ^ (s[-1] >> 62)) + i) & (2 ** 64 - 1))
        self.s, self.i = s, 312

    def __call__(self):
        if self.i == 312:
            s = self.s
            for i in range(312):
                x = (s[i] & 0xFFFFFFFF80000000) | (s[(i + 1) % 312] & 0x7FFFFFFF)
                s[i] = s[(i + 156) % 312] ^ (x >> 1) ^ (0xB5026F5AA96619E9 if x & 1 else 0)
            self.i = 0
        x = self.s[self.i]
        self.i += 1
        x ^= (x >> 29) & 0x5555555555555555
        x ^= (x << 17) & 0x71D67FFFEDA60000
        x ^= (x << 37) & 0xFFF7EEE000000000
        return x ^ (x >> 43)


def _exact_train(case, seed):
    x, y, params, norm = _samples(case, seed)
    norm = torch.tensor(norm, device="cuda").double()
    x = ((x.double() - norm[:8, None]) / norm[8:, None]).T.contiguous()
    y = y.double()
    n, batch = case["n"], case["batch"]
    perm, rng = list(range(n)), _MT64(1007)
    for k in range(n - 1, 0, -1):
        r = rng() % (k + 1)
        perm[k], perm[r] = perm[r], perm[k]
    perm = torch.tensor(perm, device="cuda")
    th = torch.tensor(params, device="cuda").double()
    m, v, total = torch.zeros_like(th), torch.zeros_like(th), 0.0
    for t, s in enumerate(range(0, n, batch), 1):
        i = perm[s:s + batch]
        p = th.clone().requires_grad_(True)
        loss = torch.nn.functional.binary_cross_entropy_with_logits(_logit(p, x[i]), y[i])
        g, = torch.autograd.grad(loss, p)
        total += float(loss.detach()) * len(i)
        m, v = 0.9 * m + 0.1 * g, 0.999 * v + 0.001 * g * g
        th = th - 1e-3 * (m / (1 - 0.9 ** t)) / ((v / (1 - 0.999 ** t)).sqrt() + 1e-8)
    return dict(params=th, loss=total / n)


def _compact(f, e):
    """The compact state (own-set populations, tile row by tile row) as deviations f / w - rho0."""
    ny, nx = f.region_map.shape
    nt = -(-nx // TILE)
    high = torch.nn.functional.pad(e.map, (0, nt * TILE - nx)).view(ny, nt, TILE)[:, :, 0]
    out = []
    for s in (0, 1):
        d = torch.nn.functional.pad(e.f[s] / e.sets[s][3] - f.rho0, (0, nt * TILE - nx)).view(-1, ny, nt, TILE)
        out.append(d[:, high if s else ~high].flatten())
    return torch.cat(out)


def exact(case, seed):
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    kind = case["kind"]
    if kind == "train":
        return _exact_train(case, seed)
    if kind == "stream":
        return _exact_box(_box(case, seed), case, dev)
    if kind == "batch":
        return _Exact(_sweep(case, seed), dev).step(case["steps"]).fields()[:3].flatten(1)
    f = _flow(case, seed)
    e = _Exact([f], dev)
    if kind == "host":
        return _compact(f, e.step(HOST_STEPS + 1))
    if kind == "place":
        feat = _exact_features(f, e.step(PLACE_STEPS).fields())
        params, norm = _network(seed)
        th = torch.tensor(params, device=dev).bfloat16().double()   # the weights inference runs with
        nm = torch.tensor(norm, device=dev).double()
        return dict(features=feat, p=torch.sigmoid(_logit(th, ((feat.flatten(1) - nm[:8, None]) / nm[8:, None]).T)))
    m = e.step(case["steps"]).fields()
    if not case.get("monitor"):
        return m
    # the first reduction compares with u = 0: its residual is 1
    return dict(fields=m, mass=float(m[0].sum()), residual=1.0, nonfinite=0, step=case["steps"])
