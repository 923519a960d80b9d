"""The work that users of this library have it do, as cases that can be timed.

Each case goes through the public binding: particle sets made from device
arrays, advanced, and read back into device arrays; the surrogate network's
inference, gradient and checked run.  Inputs are synthetic and made on the GPU
from the seed: a k^-3 random streamfunction field like the benchmark's on the
global grids (1/4 degree x 50 levels, 1/12 degree surface), the Stommel gyre
and the flow around a peninsula.  ``exact`` repeats a case in FP64 with plain
torch operations.

Positions held in FP32 are returned as FP32 (the read-back call gives them as
FP64); positions of the FP64 and the cell form as FP64.  Where the run
re-sorts the particles they are returned in the order of their ids.  Releases
on a periodic axis leave a few degrees around its seam free, so that no
returned longitude jumps by a whole turn when it is rounded differently.
"""
import math

import numpy as np
import torch

import paper_1707_05163_gb300 as pg
from paper_1707_05163_gb300 import api

DAY = 86400.0
DEG_M = 1852.0 * 60.0            # metres per degree
EARTH_R = DEG_M * 180.0 / math.pi
DEV = "cuda"

# ------------------------------------------------------------------- cases --


def listed():
    return [
        # the paper's own timing, its smallest use: 100 particles around a
        # peninsula, 20 h of 30-second RK4 steps, everything at its default
        dict(name="peninsula_100", kind="release", field="peninsula", storage="f32", pos="f32",
             n=100, scheme="rk4", dt=30.0, steps=2400, kh=0.0, w=0.0, block=0, resort=0, chunk=0),
        # the FP64 form on the benchmark's gyre: 10,000 particles, 30 days of
        # hourly steps
        dict(name="gyre_f64", kind="release", field="gyre", storage="f64", pos="f64",
             n=10_000, scheme="rk4", dt=3600.0, steps=720, kh=0.0, w=0.0, block=0, resort=0,
             chunk=0),
        # the headline workload for two of its days: 10M particles in the
        # global 3-D field, one Morton sort, the benchmark's tuning
        dict(name="global3d_10M", kind="release", field="global3d", nt=6, storage="f32", pos="f32",
             n=10_000_000, scheme="rk4", dt=1800.0, steps=96, kh=0.0, w=0.0, block=128,
             resort=1440, chunk=1440),
        # an ordinary release in the 3-D field, untuned, a ragged count,
        # drifting and sinking (plastic, plankton): backward in time
        dict(name="global3d_ragged", kind="release", field="global3d", nt=6, storage="f32",
             pos="f32", n=333_667, scheme="rk4", dt=-1200.0, steps=144, kh=10.0, w=20.0 / DAY,
             block=0, resort=0, chunk=0),
        # the precision form: cell index + offset on the 1/12-degree surface
        # field in FP16, Brownian motion
        dict(name="surface12_cell_f16", kind="release", field="surface12", nt=4, storage="f16",
             pos="cell", n=5_000_000, scheme="rk4", dt=3600.0, steps=48, kh=10.0, w=0.0,
             block=128, resort=288, chunk=288),
        # the same flow in plain FP32 positions and storage
        dict(name="surface12_f32", kind="release", field="surface12", nt=4, storage="f32",
             pos="f32", n=1_234_567, scheme="rk4", dt=3600.0, steps=48, kh=10.0, w=0.0,
             block=128, resort=288, chunk=288),
        # adaptive steps on the 3-D field, 10 m tolerance
        dict(name="rkf45_200k", kind="release", field="global3d", nt=6, storage="f32", pos="f32",
             n=200_001, scheme="rkf45", dt=1800.0, steps=96, kh=0.0, w=0.0, block=128, resort=0,
             chunk=0, tol=10.0),
        # the worked example: rise to the dwelling depth, live there, sample
        # temperature, daily indexed records; backward in 5-minute steps
        dict(name="example_records", kind="records", nt=6, n=100_000, dt=-300.0, days=9,
             depth=1050.0, max_age_days=3.5),
        # many releases of uneven size and step in one batched call
        dict(name="batch_24", kind="batch", nt=6, releases=24, n_lo=1_000, n_hi=200_000, days=4,
             block=64, resort=4),
        # one inference call of the surrogate network
        dict(name="mlp_forward_1M", kind="mlp_forward", rows=1_000_003, engine=1),
        # one gradient of a training batch
        dict(name="mlp_grad_16k", kind="mlp_grad", rows=16_384, engine=1),
        # the surrogate form: ten network steps, each fifth checked by RK4
        dict(name="surrogate_1M", kind="surrogate", nt=6, n=1_000_000, nsteps=10, check=5,
             threshold=0.5, dt=1800.0, resort=1440),
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["global3d", "global3d", "surface", "gyre", "peninsula", "rkf45", "records",
                       "batch", "mlp_forward", "mlp_grad", "surrogate"])
    tune = rng.choice([(0, 0, 0), (128, 1440, 1440), (128, 288, 288), (64, 48, 96)])
    tune = dict(block=tune[0], resort=tune[1], chunk=tune[2])
    if kind == "global3d":
        n = _logint(rng, 100, 4_000_000)
        return dict(kind="release", field="global3d", nt=6, storage=rng.choice(["f32", "f32", "f16"]),
                    pos="f32", n=n, scheme=rng.choice(["rk4", "rk4", "euler"]),
                    dt=rng.choice([1800.0, 600.0, 3600.0, -1800.0]),
                    steps=rng.randint(24, 144 if n > 500_000 else 288),
                    kh=rng.choice([0.0, 0.0, rng.uniform(1.0, 100.0)]),
                    w=rng.choice([0.0, rng.uniform(1.0, 100.0) / DAY]), **tune)
    if kind == "surface":
        return dict(kind="release", field="surface12", nt=4,
                    storage=rng.choice(["f32", "f16", "bf16"]), pos=rng.choice(["f32", "cell"]),
                    n=_logint(rng, 1_000, 4_000_000), scheme="rk4", dt=3600.0,
                    steps=rng.randint(24, 60), kh=rng.choice([0.0, 10.0]), w=0.0, **tune)
    if kind == "gyre":
        return dict(kind="release", field="gyre", storage="f64", pos="f64",
                    n=_logint(rng, 100, 40_000), scheme=rng.choice(["rk4", "euler"]), dt=3600.0,
                    steps=rng.randint(100, 720), kh=0.0, w=0.0, block=0, resort=0, chunk=0)
    if kind == "peninsula":
        return dict(kind="release", field="peninsula", storage="f32", pos="f32",
                    n=_logint(rng, 100, 20_000), scheme=rng.choice(["rk4", "euler"]),
                    dt=rng.choice([30.0, 60.0, 300.0]), steps=rng.randint(120, 240) * 2, kh=0.0,
                    w=0.0, block=0, resort=0, chunk=0)
    if kind == "rkf45":
        return dict(kind="release", field="global3d", nt=6, storage="f32", pos="f32",
                    n=_logint(rng, 1_000, 500_000), scheme="rkf45", dt=1800.0,
                    steps=rng.randint(24, 96), kh=0.0, w=0.0, tol=rng.choice([3.0, 10.0]), **tune)
    if kind == "records":
        # every particle dies in the last day, so each record has all of them
        days, rise = rng.randint(4, 9), rng.randint(1, 3)
        return dict(kind="records", nt=6, n=_logint(rng, 1_000, 200_000), dt=-300.0, days=days,
                    depth=50.0 + 200.0 * rise, max_age_days=days - rise - 0.5)
    if kind == "batch":
        return dict(kind="batch", nt=6, releases=rng.randint(4, 40), n_lo=1_000,
                    n_hi=_logint(rng, 20_000, 200_000), days=rng.randint(2, 5),
                    block=rng.choice([64, 128]), resort=rng.choice([0, 1, 4]))
    if kind == "mlp_forward":
        return dict(kind="mlp_forward", rows=_logint(rng, 100, 4_000_000),
                    engine=rng.choice([1, 1, 1, 2, 0]))
    if kind == "mlp_grad":
        return dict(kind="mlp_grad", rows=32 * _logint(rng, 8, 2_048),
                    engine=rng.choice([1, 1, 1, 0]))
    return dict(kind="surrogate", nt=6, n=_logint(rng, 1_000, 1_000_000), nsteps=rng.randint(1, 10),
                check=5, threshold=0.5, dt=1800.0, resort=rng.choice([0, 1440]))


# ------------------------------------------------------------------ fields --


def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) * 7919 + 17)
    return g


def _uniform(g, n, lo, hi):
    """FP64 values that FP32 holds exactly."""
    return (torch.rand(n, generator=g, device=DEV, dtype=torch.float64) * (hi - lo) + lo).float().double()


class Field:
    """Axes (numpy FP64), snapshot times and the snapshots as device arrays
    [nf, nz, ny, nx], made one at a time."""

    def __init__(self, lon, lat, depth, spherical, periodic, times, period, nf, snapshot):
        self.lon, self.lat, self.depth = lon, lat, depth
        self.spherical, self.periodic = spherical, periodic
        self.times, self.period, self.nf, self.snapshot = times, period, nf, snapshot


def _steady(lon, lat, u, v, dtype):
    data = torch.stack([u, v])[:, None].to(dtype).contiguous()
    return Field(lon, lat, np.zeros(1), False, False, np.zeros(1), 0.0, 2, lambda s: data)


def _gyre():
    """Stommel gyre on a flat 1000 km square, 201 x 201 nodes."""
    L, eps, psi0 = 1.0e6, 5.0e4, 1.0e5
    ax = np.linspace(0.0, L, 201)
    x = torch.tensor(ax, device=DEV)[None, :]
    y = torch.tensor(ax, device=DEV)[:, None]
    u = -psi0 * math.pi / L * torch.cos(math.pi * y / L) * (1.0 - x / L - torch.exp(-x / eps))
    v = psi0 * torch.sin(math.pi * y / L) * (-1.0 / L + torch.exp(-x / eps) / eps)
    return _steady(ax, ax, u, v, torch.float64)


def _peninsula():
    """Potential flow past a semicircular peninsula: 100 km x 50 km, 1 km."""
    x0, R, U = 5.0e4, 1.6e4, 1.0
    lon, lat = np.linspace(0.0, 1.0e5, 101), np.linspace(0.0, 5.0e4, 51)
    x = torch.tensor(lon, device=DEV)[None, :] - x0
    y = torch.tensor(lat, device=DEV)[:, None]
    r2 = (x * x + y * y).clamp(min=1.0)
    land = r2 < R * R
    u = U * (1.0 - R * R * (x * x - y * y) / r2 ** 2)
    v = -2.0 * U * R * R * x * y / r2 ** 2
    return _steady(lon, lat, u.masked_fill(land, 0.0), v.masked_fill(land, 0.0), torch.float32)


def _global(seed, nx, ny, nz, nt):
    """Global field of the benchmark's recipe: per snapshot a random-phase
    streamfunction with amplitude k^-3 (k <= 90), 0.3 m/s surface rms,
    exp(-z / 1000 m); W independent, 1e-4 m/s, zero at top and bottom;
    daily snapshots, exactly periodic."""
    lon = np.arange(nx) * (360.0 / nx)
    lat = -90.0 + (np.arange(ny) + 0.5) * (180.0 / ny)
    depth = 5.0 * 1000.0 ** (np.arange(nz) / (nz - 1)) if nz > 1 else np.zeros(1)
    g = _gen(seed)
    ky = torch.fft.fftfreq(ny, 1.0 / ny, device=DEV, dtype=torch.float64)[:, None]
    kx = torch.fft.rfftfreq(nx, 1.0 / nx, device=DEV, dtype=torch.float64)[None, :]
    k = torch.hypot(kx, ky)
    amp = torch.where((k >= 1) & (k <= 90), k.clamp(min=1.0) ** -3.0, torch.zeros_like(k))
    phase = [torch.rand(amp.shape, generator=g, device=DEV, dtype=torch.float64) * 2 * math.pi
             for _ in range(2)]
    freq = [torch.randint(0, 2, amp.shape, generator=g, device=DEV).double() * 2 - 1 for _ in range(2)]
    latr = torch.deg2rad(torch.tensor(lat, device=DEV))[:, None]
    taper, cosl = torch.cos(latr) ** 2, torch.cos(latr)
    dlam, dphi = 2 * math.pi / nx, math.pi / ny

    def psi(s, q):
        return torch.fft.irfft2(torch.polar(amp, phase[q] + 2 * math.pi * freq[q] * s / nt),
                                s=(ny, nx)) * (nx * ny) * taper

    def base(s):
        p = psi(s, 0)
        u = -torch.gradient(p, spacing=dphi, dim=0)[0] / EARTH_R
        v = (torch.roll(p, -1, 1) - torch.roll(p, 1, 1)) / (2 * dlam * EARTH_R * cosl)
        return [u, v] + ([psi(s, 1)] if nz > 1 else [])

    b0 = base(0)
    scale = [0.3 / torch.sqrt(torch.mean(b0[0] ** 2 + b0[1] ** 2))] * 2
    prof = [torch.exp(-torch.tensor(depth, device=DEV) / 1000.0) if nz > 1
            else torch.ones(1, device=DEV, dtype=torch.float64)] * 2
    if nz > 1:
        scale.append(1e-4 / torch.sqrt(torch.mean(b0[2] ** 2)))
        z = torch.tensor(depth, device=DEV)
        pw = torch.sin(math.pi * (z - z[0]) / (z[-1] - z[0]))
        pw[0] = pw[-1] = 0.0
        prof.append(pw)

    def snapshot(s):
        return torch.stack([((b * c)[None].float() * p.float()[:, None, None])
                            for b, c, p in zip(base(s), scale, prof)])

    return Field(lon, lat, depth, True, True, np.arange(nt) * DAY, nt * DAY, len(prof), snapshot)


def _field(case, seed):
    f = case.get("field", "global3d")
    if f == "gyre":
        return _gyre()
    if f == "peninsula":
        return _peninsula()
    if f == "surface12":
        return _global(seed, 4320, 2160, 1, case["nt"])
    return _global(seed, 1440, 720, 50, case["nt"])


def _fieldset(F, storage):
    fs = pg.FieldSet(F.lon, F.lat, F.depth if len(F.depth) > 1 else None,
                     mesh="spherical" if F.spherical else "flat", periodic_lon=F.periodic,
                     nfields=F.nf, storage=storage)
    fs.set_times(F.times, F.period)
    for s in range(len(F.times)):
        fs.load_snapshot(s, F.snapshot(s))
    return fs


def _temperature(F, s):
    """Sea temperature: warm surface, colder to the poles and with depth."""
    lat = torch.deg2rad(torch.tensor(F.lat, device=DEV))[None, :, None]
    z = torch.tensor(F.depth, device=DEV)[:, None, None]
    x = torch.deg2rad(torch.tensor(F.lon, device=DEV))[None, None, :]
    t = 2.0 + 26.0 * torch.cos(lat) ** 2 * torch.exp(-z / 700.0) + 0.5 * torch.sin(9 * x + 7 * lat)
    return (t + math.sin(2 * math.pi * s / len(F.times))).float()


# --------------------------------------------------------------- particles --


def _start(case, seed, n=None, salt=1):
    """Start positions (FP64 device arrays, exact in FP32)."""
    g, n = _gen(seed * 31 + salt), n or case["n"]
    f = case.get("field", "global3d")
    if f == "gyre":
        return _uniform(g, n, 0.05e6, 0.95e6), _uniform(g, n, 0.05e6, 0.95e6), None
    if f == "peninsula":
        return _uniform(g, n, 1.0e3, 8.0e3), _uniform(g, n, 2.0e3, 4.5e4), None
    if f == "surface12":
        return _uniform(g, n, 8.0, 352.0), _uniform(g, n, -80.0, 80.0), None
    return _uniform(g, n, 8.0, 352.0), _uniform(g, n, -80.0, 80.0), _uniform(g, n, 5.0, 1000.0)


def _t0(case, seed):
    """Start time: somewhere in the field's period, whole hours."""
    return 3600.0 * (seed % 24) + DAY * case["nt"] if case.get("nt") else 0.0


class State:
    pass


def _buffers(n, depth):
    b = {"lon": torch.empty(n, device=DEV, dtype=torch.float64),
         "lat": torch.empty(n, device=DEV, dtype=torch.float64),
         "status": torch.empty(n, device=DEV, dtype=torch.uint8)}
    if depth:
        b["depth"] = torch.empty(n, device=DEV, dtype=torch.float64)
    return b


def _read(ps, b, ids, f32):
    """The set's positions and status, by id where the order is not kept."""
    ps.get_into(lon=b["lon"], lat=b["lat"], depth=b.get("depth"), ids=ids, status=b["status"])
    out = {}
    for k, v in b.items():
        v = v.float() if f32 and k != "status" else v
        if ids is not None:
            v = torch.empty_like(v).index_copy_(0, ids, v)
        elif v is b[k]:
            v = v.clone()
        out[k] = v
    return out


def _releases(case):
    """Sizes, steps, durations and kernels of a batch."""
    r = np.random.default_rng([case["releases"], case["n_hi"], case["days"]])
    out = []
    for q in range(case["releases"]):
        n = int(round(math.exp(r.uniform(math.log(case["n_lo"]), math.log(case["n_hi"])))))
        dt = float(r.choice([600.0, 900.0, 1200.0, 1800.0, 2700.0, 3600.0, 5400.0, 7200.0]))
        days = float(r.uniform(1.0, case["days"]))
        beh = int(r.integers(0, 3))
        out.append(dict(n=n, dt=dt, runtime=math.floor(days * DAY / dt) * dt,
                        kh=float(np.exp(r.uniform(0.0, math.log(100.0)))) if beh == 1 else 0.0,
                        w=float(np.exp(r.uniform(0.0, math.log(100.0)))) / DAY if beh == 2 else 0.0))
    return out


def _kernel(scheme, kh, w, more=()):
    beh = (("brownian",) if kh else ()) + (("sink",) if w else ()) + tuple(more)
    return pg.Kernel(scheme, beh, kh=kh, w_sink=w if not more else None)


def _net_params(net, seed):
    """Weights of a linear flow map in the network's layout, as a stand-in for
    trained ones: the displacement the velocities at the cell's four corners
    give over a day, carried through the layers by the pairs GELU(x) -
    GELU(-x) = x, with small random weights in the remaining units."""
    r = np.random.default_rng(seed * 13 + 3)
    n_in, W = 37, 256
    dims = [(64, W), (W, W), (W, W), (W, W), (W, 64)]
    parts = []
    for l, (din, dout) in enumerate(dims):
        w = np.zeros((dout, din), np.float32)
        b = np.zeros(dout, np.float32)
        if l == 0:
            w[8:W, :n_in] = r.normal(0, 0.05, (W - 8, n_in))
            for c in range(2):
                row = np.zeros(din, np.float32)
                for q in (5, 6, 9, 10):                  # 4 x 4 stencil, inner corners
                    row[5 + 2 * q + c] = 0.25 * 0.3 * DAY / (DEG_M * 0.25)
                w[2 * c], w[2 * c + 1] = row, -row
        elif l < 4:
            w[8:W, 8:W] = r.normal(0, 0.05, (W - 8, W - 8))
            for c in range(2):
                w[2 * c, 2 * c], w[2 * c, 2 * c + 1] = 1.0, -1.0
                w[2 * c + 1, 2 * c], w[2 * c + 1, 2 * c + 1] = -1.0, 1.0
        else:
            w[:3, 8:W] = r.normal(0, 0.002, (3, W - 8))
            for c in range(2):
                w[c, 2 * c], w[c, 2 * c + 1] = 1.0, -1.0
        if l < 4:
            b[8:W] = r.normal(0, 0.02, W - 8)
        parts += [w.ravel(), b]
    return np.concatenate(parts)


def _random_params(seed):
    """Weights as a training run meets them: He-scaled, small output layer."""
    r = np.random.default_rng(seed * 17 + 5)
    parts = []
    for l, (din, rin, dout, rout) in enumerate([(64, 37, 256, 256)] + [(256, 256, 256, 256)] * 3 +
                                               [(256, 256, 64, 3)]):
        w = np.zeros((dout, din), np.float32)
        w[:rout, :rin] = r.uniform(-1, 1, (rout, rin)) * math.sqrt(6.0 / rin) * (0.1 if l == 4 else 1.0)
        b = np.zeros(dout, np.float32)
        b[:rout] = r.normal(0, 0.05, rout)
        parts += [w.ravel(), b]
    return np.concatenate(parts)


def _rows(case, seed):
    g = _gen(seed)
    x = torch.randn(case["rows"], 37, generator=g, device=DEV)
    return x, torch.randn(case["rows"], 3, generator=g, device=DEV)


def prepare(case, seed):
    s = State()
    s.case, s.seed = case, seed
    kind = case["kind"]
    if kind in ("mlp_forward", "mlp_grad"):
        s.net = pg.MLP(37, 256, 4, 3, seed=1)
        s.net.set_engine(case["engine"])
        s.net.set_params(_random_params(seed))
        s.x, s.t = _rows(case, seed)
        s.y = torch.empty(case["rows"], 3, device=DEV)
        return s
    F = _field(case, seed)
    s.fs = _fieldset(F, case.get("storage", "f32"))
    s.t0 = _t0(case, seed)
    if kind == "batch":
        s.rel = _releases(case)
        s.start = [_start(case, seed, r["n"], 100 + q) for q, r in enumerate(s.rel)]
        s.kernels = [_kernel("rk4", r["kh"], r["w"]) for r in s.rel]
        s.ids = [torch.empty(r["n"], device=DEV, dtype=torch.int64) for r in s.rel]
        s.buf = [_buffers(r["n"], True) for r in s.rel]
        return s
    if kind == "records":
        g = _gen(seed * 31 + 1)
        s.start = (_uniform(g, case["n"], 15.3, 19.3), _uniform(g, case["n"], -36.7, -32.7),
                   torch.full((case["n"],), case["depth"], device=DEV, dtype=torch.float64).float().double())
        s.fs.add_scalar("temperature")
        for q in range(case["nt"]):
            s.fs.load_scalar(0, q, _temperature(F, q))
        s.fs.add_constant("w_sink", 200.0 / DAY)
        s.fs.add_constant("dwelling_depth", 50.0)
        s.fs.add_constant("max_age", case["max_age_days"] * DAY)
        s.kernel = _kernel("rk4", 0.0, 0.0, ("settle", "age", "sample"))
        s.t0 += 2 * case["nt"] * DAY
        return s
    s.start = _start(case, seed)
    s.buf = _buffers(case["n"], s.start[2] is not None)
    s.ids = torch.empty(case["n"], device=DEV, dtype=torch.int64) if case["resort"] else None
    if kind == "surrogate":
        s.net = pg.MLP(37, 256, 4, 3, seed=1)
        s.net.set_engine(1)
        s.net.set_params(_net_params(s.net, seed))
        s.kernel = _kernel("rk4", 0.0, 0.0)
        return s
    if case["scheme"] == "rkf45":
        s.fs.add_constant("rkf45_tol", case["tol"])
        s.fs.add_constant("rkf45_min_dt", 60.0)
        s.fs.add_constant("rkf45_max_dt", 7200.0)
    s.kernel = _kernel(case["scheme"], case["kh"], case["w"])
    return s


def run(s):
    case, kind = s.case, s.case["kind"]
    if kind == "mlp_forward":
        return {"y": s.net.forward(s.x, out=s.y)}
    if kind == "mlp_grad":
        loss, g = s.net.grad(s.x, s.t)
        return {"loss": loss, "grad": g}
    if kind == "batch":
        ps = [pg.ParticleSet(s.fs, *p, t0=s.t0, pos="f32", seed=q) for q, p in enumerate(s.start)]
        pg.execute_batch(ps, s.kernels, [r["runtime"] for r in s.rel], [r["dt"] for r in s.rel],
                         tune=(case["block"], case["resort"]))
        outs = [_read(p, b, i, True) for p, b, i in zip(ps, s.buf, s.ids)]
        for p in ps:
            p.destroy()
        return {k: torch.cat([o[k] for o in outs]) for k in outs[0]}
    lon, lat, dep = s.start
    if kind == "records":
        rows = []
        ps = pg.ParticleSet(s.fs, lon, lat, dep, t0=s.t0, pos="f32")
        ps.execute_records(s.kernel, case["days"] * DAY, case["dt"], DAY,
                           lambda t, r: rows.append(r))
        ps.destroy()
        out = {k: np.concatenate([r[k] for r in rows]) for k in ("id", "lon", "lat", "depth", "age")}
        out["id"] = out["id"].astype(np.int64)
        for k in ("lon", "lat", "depth"):
            out[k] = out[k].astype(np.float32)
        out["status"] = np.concatenate([r["status"] for r in rows])
        out["temperature"] = np.concatenate([r["vars"][0] for r in rows]).astype(np.float32)
        return out
    ps = pg.ParticleSet(s.fs, lon, lat, dep, t0=s.t0, pos=case.get("pos", "f32"), seed=s.seed)
    if kind == "surrogate":
        ps.set_tune(0, case["resort"], 0)
        st = api.surrogate_run(ps, s.net, s.kernel, nsteps=case["nsteps"], check_every=case["check"],
                               dt_check=case["dt"], threshold=case["threshold"])
        out = _read(ps, s.buf, s.ids, True)
        out["mean_check_error"] = torch.tensor(st["error_sum"] / max(1, st["checked"]),
                                               dtype=torch.float32)
    else:
        if case["block"]:
            ps.set_tune(case["block"], case["resort"], case["chunk"])
        ps.execute(s.kernel, case["steps"] * abs(case["dt"]), case["dt"])
        out = _read(ps, s.buf, s.ids, case["pos"] == "f32")
    ps.destroy()
    return out


# -------------------------------------------------------------------- work --


def work(case):
    """What a pass cannot do without: positions read and written once, the
    snapshots that the run's time spans read once (at most the corners its
    stages ask for), and the arithmetic of the interpolations."""
    kind = case["kind"]
    per_row = 2.0 * (37 * 256 + 3 * 256 * 256 + 256 * 3)
    weights = 4.0 * (37 * 256 + 3 * 256 * 256 + 256 * 3 + 4 * 256 + 3)
    if kind == "mlp_forward":
        return {"bytes": case["rows"] * 4.0 * 40 + weights, "flops": case["rows"] * per_row}
    if kind == "mlp_grad":
        return {"bytes": case["rows"] * 4.0 * 40 + 2 * weights, "flops": 3.0 * case["rows"] * per_row}
    f = case.get("field", "global3d")
    el = {"f64": 8, "f32": 4}.get(case.get("storage", "f32"), 2)
    nodes = {"gyre": 201 * 201, "peninsula": 101 * 51, "surface12": 4320 * 2160,
             "global3d": 1440 * 720 * 38}[f] * el * (3 if f == "global3d" else 2)
    stage = 110.0 if f == "global3d" else 50.0

    def snaps(span):
        return 1 if not case.get("nt") else min(case["nt"], int(span / DAY) + 2)

    if kind == "batch":
        rel = _releases(case)
        n = sum(r["n"] for r in rel)
        steps = sum(r["n"] * r["runtime"] / r["dt"] for r in rel)
        return {"bytes": n * 57.0 + min(nodes * snaps(case["days"] * DAY), steps * 768.0),
                "flops": steps * (4 * stage + 10)}
    n = case["n"]
    if kind == "records":
        steps = n * (min(case["days"] * DAY, (case["depth"] - 50.0) / 200.0 * DAY +
                         case["max_age_days"] * DAY) / -case["dt"])
        return {"bytes": n * (24.0 + 49.0 * case["days"]) + 0.01 * nodes * snaps(case["days"] * DAY),
                "flops": steps * (4 * stage + 20)}
    if kind == "surrogate":
        rk = n * (DAY / case["dt"]) * math.ceil(case["nsteps"] / case["check"])
        return {"bytes": n * 57.0 + min(nodes * snaps(case["nsteps"] * DAY), n * 512.0 * case["nsteps"]),
                "flops": rk * (4 * stage + 10) + n * case["nsteps"] * per_row}
    stages = {"rk4": 4, "euler": 1, "rkf45": 6}[case["scheme"]]
    steps = case["steps"] if case["scheme"] != "rkf45" else case["steps"] / 4.0
    pos = 24 + 25 if f == "global3d" else 16 + 17
    corners = (48 if f == "global3d" else 16) * el
    return {"bytes": n * float(pos) + min(float(nodes) * snaps(case["steps"] * abs(case["dt"])),
                                          float(n) * steps * corners),
            "flops": n * steps * (stages * stage + 10.0 + (60.0 if case["kh"] else 0.0))}


# ------------------------------------------------------------------- exact --


class Exact:
    """A field for FP64 evaluation: all snapshots in one array."""

    def __init__(self, F, storage):
        data = []
        for s in range(len(F.times)):
            d = F.snapshot(s)
            if storage in ("f16", "bf16"):    # codes with one FP32 scale per plane
                sc = (d.float().abs().amax(dim=(1, 2, 3), keepdim=True) / 32752.0)
                half = torch.float16 if storage == "f16" else torch.bfloat16
                d = (d.float() / sc).to(half).float() * sc
            data.append(d)
        self.data = torch.stack(data)
        self.flat = self.data.view(-1)
        self.nt, self.nf, self.nz, self.ny, self.nx = self.data.shape
        dt = torch.float64
        self.ax = [torch.tensor(a, device=DEV, dtype=dt) for a in (F.lon, F.lat, F.depth)]
        self.times = torch.tensor(F.times, device=DEV, dtype=dt)
        self.period, self.sph, self.per = F.period, F.spherical, F.periodic

    def wrap(self, lon):
        x0 = self.ax[0][0]
        return x0 + torch.remainder(lon - x0, 360.0) if self.per else lon

    def outside(self, lon, lat, dep):
        """0, or the status of a position outside the domain."""
        bad = ~((lat >= self.ax[1][0]) & (lat <= self.ax[1][-1]))
        if not self.per:
            bad = bad | ~((lon >= self.ax[0][0]) & (lon <= self.ax[0][-1]))
        st = bad.to(torch.uint8)
        if self.nz > 1:
            deep = ~((dep >= self.ax[2][0]) & (dep <= self.ax[2][-1]))
            st = torch.where((st == 0) & deep, torch.full_like(st, 2), st)
        return st

    def cell(self, a, p):
        x = self.ax[a]
        i = (torch.searchsorted(x, p, right=True) - 1).clamp(0, len(x) - 2)
        return i, (p - x[i]) / (x[i + 1] - x[i])

    def interval(self, t):
        if self.nt == 1:
            return torch.zeros_like(t, dtype=torch.int64), torch.zeros_like(t, dtype=torch.int64), torch.zeros_like(t)
        T = self.times
        r = torch.remainder(t - T[0], self.period) + T[0]
        s0 = (torch.searchsorted(T, r, right=True) - 1).clamp(0, self.nt - 1)
        s1 = torch.where(s0 + 1 < self.nt, s0 + 1, torch.zeros_like(s0))
        end = torch.where(s0 + 1 < self.nt, T[s1], T[0] + self.period)
        return s0, s1, (r - T[s0]) / (end - T[s0])

    def locate(self, lon, lat, dep):
        lon = self.wrap(lon)
        i, xi = self.cell(0, lon)
        i1 = i + 1
        if self.per:
            last = lon >= self.ax[0][-1]
            gap = self.ax[0][0] + 360.0 - self.ax[0][-1]
            i = torch.where(last, torch.full_like(i, self.nx - 1), i)
            i1 = torch.where(last, torch.zeros_like(i), i1)
            xi = torch.where(last, (lon - self.ax[0][-1]) / gap, xi)
        j, eta = self.cell(1, lat)
        if self.nz > 1:
            k, zeta = self.cell(2, dep)
        else:
            k, zeta = torch.zeros_like(i), torch.zeros_like(lon)
        return i, i1, xi, j, eta, k, zeta

    def sample(self, t, lon, lat, dep, flat=None, nf=None):
        """Field values at positions inside the domain (linear in space and time)."""
        flat, nf = (self.flat, self.nf) if flat is None else (flat, nf)
        i, i1, xi, j, eta, k, zeta = self.locate(lon, lat, dep)
        s0, s1, tau = self.interval(t)
        out = []
        for f in range(nf):
            v = 0.0
            for s, ws in ((s0, 1.0 - tau), (s1, tau)):
                if self.nt == 1 and s is s1:
                    continue
                for kk in range(2 if self.nz > 1 else 1):
                    wz = (zeta if kk else 1.0 - zeta) if self.nz > 1 else 1.0
                    row = ((s * nf + f) * self.nz + k + kk) * self.ny
                    for jj in range(2):
                        wy = eta if jj else 1.0 - eta
                        b = (row + j + jj) * self.nx
                        v = v + ws * wz * wy * ((1.0 - xi) * flat[b + i].double() +
                                                xi * flat[b + i1].double())
            out.append(v)
        return out

    def velocity(self, t, lon, lat, dep):
        """(rates in position units, status of positions outside)."""
        st = self.outside(lon, lat, dep)
        lon = torch.where(st == 0, lon, self.ax[0][0])
        lat = torch.where(st == 0, lat, self.ax[1][0])
        dep = torch.where(st == 0, dep, self.ax[2][0])
        v = self.sample(t, lon, lat, dep)
        if len(v) == 2:
            v.append(torch.zeros_like(lon))
        if self.sph:
            v[0] = v[0] / (DEG_M * torch.cos(torch.deg2rad(lat)))
            v[1] = v[1] / DEG_M
        return v, st


def _normals(seed, ids, step):
    """Standard normal pairs of Philox4x32-10 with counter (id, step)."""
    m32 = 0xFFFFFFFF
    c = [ids & m32, ids >> 32, step, torch.zeros_like(ids)]
    k = [seed & m32, seed >> 32]
    for r in range(10):
        if r:
            k = [(k[0] + 0x9E3779B9) & m32, (k[1] + 0xBB67AE85) & m32]
        p0, p1 = c[0] * 0xD2511F53, c[2] * 0xCD9E8D57
        c = [((p1 >> 32) & m32) ^ c[1] ^ k[0], p1 & m32, ((p0 >> 32) & m32) ^ c[3] ^ k[1], p0 & m32]
    m1 = ((c[0] >> 5) << 26) | (c[1] >> 6)
    m2 = ((c[2] >> 5) << 26) | (c[3] >> 6)
    u1, u2 = (m1.double() + 1.0) * 2.0 ** -53, m2.double() * 2.0 ** -53
    rad = torch.sqrt(-2.0 * torch.log(u1))
    return rad * torch.cos(2 * math.pi * u2), rad * torch.sin(2 * math.pi * u2)


class Advect:
    """Particles in FP64; dt, kh, w and end time per particle."""

    def __init__(self, E, start, t0, dt, kh=0.0, w=0.0, seed=0, ids=None, status=None):
        full = lambda v: v if isinstance(v, torch.Tensor) else torch.full_like(start[0], float(v))  # noqa: E731
        self.E = E
        self.lon, self.lat = start[0].clone(), start[1].clone()
        self.dep = start[2].clone() if start[2] is not None else torch.zeros_like(self.lon)
        self.t, self.dt, self.kh, self.w = full(t0).clone(), full(dt), full(kh), full(w)
        n = len(self.lon)
        self.ids = torch.arange(n, device=DEV) if ids is None else ids
        self.seed = seed if isinstance(seed, torch.Tensor) else torch.full((n,), seed, device=DEV)
        self.step = torch.zeros(n, device=DEV, dtype=torch.int64)
        self.status = torch.zeros(n, device=DEV, dtype=torch.uint8) if status is None else status.clone()
        self.noise, self.age, self.settle = bool((self.kh > 0).any()), None, None

    def stages(self, h, weights_a, times_c):
        """Slopes of an explicit scheme from the current state."""
        ks, st = [], torch.zeros_like(self.status)
        for a, c in zip(weights_a, times_c):
            p = [self.lon, self.lat, self.dep]
            for q, aq in enumerate(a):
                if aq:
                    p = [x + h * aq * k for x, k in zip(p, ks[q])]
            v, s = self.E.velocity(self.t + c * h, *p)
            st = torch.where(st == 0, s, st)
            ks.append(v)
        return ks, st

    def finish(self, new, h, on, st):
        """Behaviours, wrap, domain test; moves the particles of `on`."""
        lon, lat, dep = new
        if self.noise:
            n1, n2 = _normals(self.seed, self.ids, self.step)
            sig = torch.sqrt(2.0 * self.kh * h.abs())
            if self.E.sph:
                lon = lon + sig * n1 / (DEG_M * torch.cos(torch.deg2rad(lat)))
                lat = lat + sig * n2 / DEG_M
            else:
                lon, lat = lon + sig * n1, lat + sig * n2
        dwell = None
        if self.settle is None:
            dep = dep + self.w * h
        else:
            zd, ws = self.settle
            dwell = self.dep == zd
            moved = dep + ws * h
            moved = torch.where((self.dep - zd) * (moved - zd) <= 0, torch.full_like(moved, zd), moved)
            dep = torch.where(dwell, torch.full_like(dep, zd), moved)
        lon = self.E.wrap(lon)
        st = torch.where(st == 0, self.E.outside(lon, lat, dep), st)
        go = on & (st == 0)
        self.status = torch.where(on & (st != 0), st, self.status)
        self.lon = torch.where(go, lon, self.lon)
        self.lat = torch.where(go, lat, self.lat)
        self.dep = torch.where(go, dep, self.dep)
        self.t = torch.where(go, self.t + h, self.t)
        self.step = self.step + go
        if self.age is not None:
            self.age = torch.where(go & dwell, self.age + h.abs(), self.age)
            self.status = torch.where(go & (self.age >= self.max_age),
                                      torch.full_like(self.status, 4), self.status)
        return go

    def on(self, t_end):
        return (self.status == 0) & (torch.sign(self.dt) * (t_end - self.t) > 0)

    def one_step(self, t_end, scheme):
        on = self.on(t_end)
        left = t_end - self.t
        h = torch.where(left.abs() < self.dt.abs(), left, self.dt)
        h = torch.where(on, h, self.dt)
        if scheme == "euler":
            ks, st = self.stages(h, [[]], [0.0])
            new = [x + h * k for x, k in zip((self.lon, self.lat, self.dep), ks[0])]
        else:
            ks, st = self.stages(h, [[], [0.5], [0.0, 0.5], [0.0, 0.0, 1.0]], [0.0, 0.5, 0.5, 1.0])
            new = [x + (a + 2 * b + 2 * c + d) / 6 * h for x, a, b, c, d in
                   zip((self.lon, self.lat, self.dep), *ks)]
        self.finish(new, h, on, st)

    def run(self, t_end, scheme="rk4"):
        """All steps to t_end; many steps as replays of one captured graph."""
        n = int(((t_end - self.t) / self.dt).max().clamp(min=0.0).ceil())
        if n < 8:
            for _ in range(n):
                self.one_step(t_end, scheme)
            return
        self.one_step(t_end, scheme)
        names = ["lon", "lat", "dep", "t", "step", "status"] + (["age"] if self.age is not None else [])
        held = {k: getattr(self, k).clone() for k in names}
        for k in names:
            setattr(self, k, held[k])
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            self.one_step(t_end, scheme)
            for k in names:
                held[k].copy_(getattr(self, k))
        for k in names:
            setattr(self, k, held[k])
        for _ in range(n - 1):
            graph.replay()
        torch.cuda.synchronize()

    def run_rkf45(self, t_end, tol, hmin, hmax):
        A = [[], [1 / 4], [3 / 32, 9 / 32], [1932 / 2197, -7200 / 2197, 7296 / 2197],
             [439 / 216, -8.0, 3680 / 513, -845 / 4104],
             [-8 / 27, 2.0, -3544 / 2565, 1859 / 4104, -11 / 40]]
        C = [0.0, 1 / 4, 3 / 8, 12 / 13, 1.0, 1 / 2]
        B4 = [25 / 216, 0.0, 1408 / 2565, 2197 / 4104, -1 / 5, 0.0]
        B5 = [16 / 135, 0.0, 6656 / 12825, 28561 / 56430, -9 / 50, 2 / 55]
        sg, hp = torch.sign(self.dt), self.dt.clone()
        while True:
            on = self.on(t_end)
            if not bool(on.any()):
                return
            left = t_end - self.t
            clip = left.abs() < hp.abs()
            h = torch.where(clip, left, hp)
            ks, st = self.stages(h, A, C)
            x4, err = [], []
            for a, x in enumerate((self.lon, self.lat, self.dep)):
                d4 = sum(b * k[a] for b, k in zip(B4, ks))
                d5 = sum(b * k[a] for b, k in zip(B5, ks))
                x4.append(x + h * d4)
                err.append((h * (d5 - d4)).abs())
            if self.E.sph:
                err[0] = err[0] * DEG_M * torch.cos(torch.deg2rad(x4[1]))
                err[1] = err[1] * DEG_M
            e = torch.maximum(torch.maximum(err[0], err[1]), err[2])
            no = on & (st == 0) & (e > tol) & (h.abs() > hmin)
            go = self.finish(x4, h, on & ~no, st)
            hp = torch.where(no, sg * (h.abs() / 2).clamp(min=hmin), hp)
            hp = torch.where(go & ~clip & (e < tol / 10), sg * (2 * hp.abs()).clamp(max=hmax), hp)

    def out(self, E, f32):
        d = {"lon": self.lon, "lat": self.lat, "status": self.status}
        if E.nz > 1:
            d["depth"] = self.dep
        return d


def _mlp64(flat, x):
    """The network in FP64: GELU in its tanh form."""
    p, at, h = torch.tensor(flat, device=DEV, dtype=torch.float64), 0, x.double()
    h = torch.nn.functional.pad(h, (0, 64 - h.shape[1]))
    for l, (din, dout) in enumerate([(64, 256)] + [(256, 256)] * 3 + [(256, 64)]):
        w = p[at:at + din * dout].view(dout, din)
        b = p[at + din * dout:at + din * dout + dout]
        at += din * dout + dout
        h = h @ w.T + b
        if l < 4:
            h = torch.nn.functional.gelu(h, approximate="tanh")
    return h[:, :3]


def _mlp64_grad(flat, x, t):
    """Gradient of 0.5 mean_rows sum_out (y - t)^2, and the loss."""
    p = torch.tensor(flat, device=DEV, dtype=torch.float64)
    dims, at, ws = [(64, 256)] + [(256, 256)] * 3 + [(256, 64)], 0, []
    for din, dout in dims:
        ws.append((p[at:at + din * dout].view(dout, din).clone().requires_grad_(True),
                   p[at + din * dout:at + din * dout + dout].clone().requires_grad_(True)))
        at += din * dout + dout
    h = torch.nn.functional.pad(x.double(), (0, 64 - x.shape[1]))
    for l, (w, b) in enumerate(ws):
        h = h @ w.T + b
        if l < 4:
            h = torch.nn.functional.gelu(h, approximate="tanh")
    loss = 0.5 * ((h[:, :3] - t.double()) ** 2).sum() / len(x)
    loss.backward()
    # the padded rows of the last layer have no part in the loss; the library
    # gives zero for them as autograd does
    return loss.item(), torch.cat([v.grad.reshape(-1) for wb in ws for v in wb])


def _features64(E, P):
    i, i1, xi, j, eta, k, zeta = E.locate(P.lon, P.lat, P.dep)
    s0, s1, tau = E.interval(P.t)
    phase = torch.remainder(P.t - E.times[0], E.period) / E.period
    cols = [xi, eta, P.lat / 90.0, P.dep / 1000.0, phase]
    for dj in range(-1, 3):
        jj = (j + dj).clamp(0, E.ny - 1)
        for di in range(-1, 3):
            ii = torch.remainder(i + di, E.nx)
            for f in range(2):
                at = lambda s, kk: E.flat[(((s * E.nf + f) * E.nz + k + kk) * E.ny + jj) * E.nx + ii].double()  # noqa: E731
                a = at(s0, 0) * (1 - zeta) + at(s0, 1) * zeta
                b = at(s1, 0) * (1 - zeta) + at(s1, 1) * zeta
                cols.append((a * (1 - tau) + b * tau) / 0.3)
    return torch.stack(cols, 1)


def _surrogate64(case, seed, E, start, t0):
    flat = _net_params(None, seed)
    cell = 360.0 / E.nx
    P = Advect(E, start, t0, case["dt"])
    done, esum, checked = 0, 0.0, 0

    def net_step():
        y = _mlp64(flat, _features64(E, P))
        new = [P.lon + y[:, 0] * cell, P.lat + y[:, 1] * cell, P.dep + y[:, 2] * 100.0]
        P.finish(new, torch.full_like(P.t, DAY), P.status == 0, torch.zeros_like(P.status))

    def copy(Q):
        R = Advect(E, (Q.lon, Q.lat, Q.dep), Q.t, case["dt"], status=Q.status)
        return R

    while done < case["nsteps"]:
        blk = min(case["check"], case["nsteps"] - done)
        ck = copy(P)
        for _ in range(blk - 1):
            net_step()
        chk = copy(P)
        net_step()
        chk.run(chk.t + DAY)
        dl = torch.remainder(P.lon - chk.lon + 180.0, 360.0) - 180.0
        kz, _ = E.cell(2, chk.dep)
        layer = E.ax[2][kz + 1] - E.ax[2][kz]
        e = torch.maximum(torch.maximum(dl.abs(), (P.lat - chk.lat).abs()) / cell,
                          (P.dep - chk.dep).abs() / layer)
        both = (P.status == 0) & (chk.status == 0) & (ck.status == 0)
        esum += float(e[both].sum())
        checked += int(both.sum())
        rej = (ck.status == 0) & (~both | ~(e <= case["threshold"]))
        end = ck.t + blk * DAY
        ck.status = torch.where(rej, ck.status, torch.full_like(ck.status, 1))
        ck.run(end)
        for k in ("lon", "lat", "dep", "t", "status"):
            setattr(P, k, torch.where(rej, getattr(ck, k), getattr(chk, k)))
        done += blk
    out = P.out(E, True)
    out["mean_check_error"] = torch.tensor(esum / max(1, checked), dtype=torch.float64)
    return out


def exact(case, seed):
    kind = case["kind"]
    if kind == "mlp_forward":
        x, _ = _rows(case, seed)
        flat = _random_params(seed)
        return {"y": torch.cat([_mlp64(flat, c) for c in x.split(1 << 18)])}
    if kind == "mlp_grad":
        x, t = _rows(case, seed)
        loss, g = _mlp64_grad(_random_params(seed), x, t)
        return {"loss": loss, "grad": g}
    # over a few million particles the FP64 evaluation takes minutes
    if kind != "batch" and case["n"] * case.get("steps", 300) > 4.0e8:
        return None
    E = Exact(_field(case, seed), case.get("storage", "f32"))
    t0 = _t0(case, seed)
    if kind == "batch":
        rel = _releases(case)
        st = [_start(case, seed, r["n"], 100 + q) for q, r in enumerate(rel)]
        each = lambda f: torch.cat([torch.full((r["n"],), f(q, r), device=DEV, dtype=torch.float64)  # noqa: E731
                                    for q, r in enumerate(rel)])
        P = Advect(E, [torch.cat([s[a] for s in st]) for a in range(3)], t0, each(lambda q, r: r["dt"]),
                   each(lambda q, r: r["kh"]), each(lambda q, r: r["w"]),
                   torch.cat([torch.full((r["n"],), q, device=DEV) for q, r in enumerate(rel)]),
                   torch.cat([torch.arange(r["n"], device=DEV) for r in rel]))
        P.run(t0 + each(lambda q, r: r["runtime"]))
        return P.out(E, True)
    if kind == "records":
        s = _gen(seed * 31 + 1)
        n = case["n"]
        start = (_uniform(s, n, 15.3, 19.3), _uniform(s, n, -36.7, -32.7),
                 torch.full((n,), case["depth"], device=DEV, dtype=torch.float64).float().double())
        t0 += 2 * case["nt"] * DAY
        F = _field(case, seed)
        temp = torch.stack([_temperature(F, q) for q in range(case["nt"])]).view(-1)
        P = Advect(E, start, t0, case["dt"])
        P.age, P.max_age, P.settle = torch.zeros_like(P.lon), case["max_age_days"] * DAY, (50.0, 200.0 / DAY)
        rows = []
        for d in range(case["days"]):
            was = P.status == 0
            P.run(t0 - (d + 1) * DAY)
            T = E.sample(P.t, P.lon, P.lat, P.dep, temp, 1)[0]
            rows.append([v[was] for v in (P.ids, P.lon, P.lat, P.dep, P.age, P.status, T)])
        cat = [torch.cat(c) for c in zip(*rows)]
        return dict(zip(("id", "lon", "lat", "depth", "age", "status", "temperature"), cat))
    start = _start(case, seed)
    if kind == "surrogate":
        return _surrogate64(case, seed, E, start, t0)
    P = Advect(E, start, t0, case["dt"], case["kh"], case["w"], seed)
    end = t0 + case["steps"] * case["dt"]
    if case["scheme"] == "rkf45":
        P.run_rkf45(end, case["tol"], 60.0, 7200.0)
    else:
        P.run(end, case["scheme"])
    return P.out(E, True)
