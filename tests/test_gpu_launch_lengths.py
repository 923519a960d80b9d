"""FP32 results do not depend on where launches end, for steps at whole-second
times: a time on a snapshot belongs to the interval after it and a position on
a node to the cell above it (Sect. 2.3, 2.4), whichever interval and cell the
particle comes from.  The lengths used here show a difference: 25200 s (seven
hours), 41 and 47 times their FP32 reciprocals are 1 - 2^-24.

Launches of the library's own length (up to 1440 steps) are compared with
short ones, bit for bit; and particles on the last nodes of a closed domain
with the FP64 form."""
import numpy as np
import pytest

import synth
from tests.helpers import cell_error

pytestmark = pytest.mark.gpu

H = 3600.0


@pytest.fixture(scope="module")
def pg():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    import paper_1707_05163_gb300 as pg
    pg.load()
    return pg


def _same(a, b, what=""):
    for k in ("lon", "lat", "depth", "time", "step", "status"):
        np.testing.assert_array_equal(a[k], b[k], err_msg=f"{k} {what}")


@pytest.mark.parametrize("sgn", [1, -1])
@pytest.mark.parametrize("pos,storage,nz", [("f32", "f32", 1), ("f32", "f32", 3), ("cell", "f16", 1)])
def test_launches_that_start_on_snapshot_times(pg, pos, storage, nz, sgn):
    """Snapshots every seven hours, half-hour steps: launches of 14 steps start
    on snapshot times, those of 7 and of the default length also between and
    across them."""
    rng = np.random.default_rng(3)
    nx, ny, nt = 24, 13, 5
    spec = synth.FieldSpec(np.arange(nx) * 15.0, -45.0 + 7.5 * np.arange(ny),
                           np.linspace(0.0, 100.0, nz) if nz > 1 else np.zeros(1),
                           np.arange(nt) * 7 * H, rng.normal(size=(nt, 2, nz, ny, nx)) * 3.0, 1, True,
                           nt * 7 * H, 2, None)
    fs = pg.FieldSet.from_spec(spec, storage=storage)
    lon = rng.uniform(0.0, 360.0, 20_000).astype(np.float32)
    lat = rng.uniform(-30.0, 30.0, 20_000).astype(np.float32)
    dep = rng.uniform(5.0, 95.0, 20_000).astype(np.float32) if nz > 1 else None
    out = []
    for chunk in (0, 14, 7):
        ps = pg.ParticleSet(fs, lon, lat, dep, t0=nt * 7 * H, pos=pos)
        if chunk:
            ps.set_tune(block=128, resort_steps=0, chunk_steps=chunk)
        ps.execute(pg.Kernel("rk4"), 70 * 1800.0, sgn * 1800.0)
        out.append(ps.get())
    assert (out[0]["status"] == 0).mean() > 0.9
    _same(out[0], out[1], "14 steps")
    _same(out[0], out[2], "7 steps")


@pytest.mark.parametrize("sgn", [1, -1])
def test_adaptive_steps(pg, sgn):
    """RKF45 over snapshots every seven hours: trials that are rejected after a
    stage past a snapshot, steps of a few minutes and fractions of them."""
    rng = np.random.default_rng(8)
    nx, ny, nz, nt = 24, 13, 3, 5
    spec = synth.FieldSpec(np.arange(nx) * 15.0, -45.0 + 7.5 * np.arange(ny),
                           np.linspace(0.0, 100.0, nz), np.arange(nt) * 7 * H,
                           rng.normal(size=(nt, 3, nz, ny, nx)) * np.array([9.0, 9.0, 1e-4])[:, None, None, None],
                           1, True, nt * 7 * H, 3, None)
    fs = pg.FieldSet.from_spec(spec, storage="f32")
    fs.add_constant("rkf45_tol", 0.3)
    fs.add_constant("rkf45_min_dt", 50.0)
    fs.add_constant("rkf45_max_dt", 4 * H)
    lon = rng.uniform(0.0, 360.0, 20_000).astype(np.float32)
    lat = rng.uniform(-30.0, 30.0, 20_000).astype(np.float32)
    dep = rng.uniform(5.0, 95.0, 20_000).astype(np.float32)
    out = []
    for chunk in (0, 14, 5):
        ps = pg.ParticleSet(fs, lon, lat, dep, t0=2 * nt * 7 * H, pos="f32")
        ps.set_tune(block=128, resort_steps=0, chunk_steps=chunk)
        ps.execute(pg.Kernel("rkf45"), 70 * 1800.0, sgn * 1800.0)
        out.append(ps.get())
    assert (out[0]["status"] == 0).mean() > 0.8
    assert out[0]["step"][out[0]["status"] == 0].std() > 1.0
    _same(out[0], out[1], "14 steps")
    _same(out[0], out[2], "5 steps")


def test_launches_that_start_on_cell_faces(pg):
    """Longitudes near 1e7 m are whole metres in FP32 and the cells 41 m wide, so
    steps often end on a face; the latitude, near zero, shows the fraction's
    last bit."""
    rng = np.random.default_rng(4)
    nx, ny = 120, 9
    lon_ax = 1.0e7 + 41.0 * np.arange(nx)
    lat_ax = np.linspace(-1.0, 1.0, ny)
    uv = rng.normal(size=(1, 2, 1, ny, nx)) * np.array([3.0, 1e-3])[None, :, None, None, None]
    spec = synth.FieldSpec(lon_ax, lat_ax, np.zeros(1), np.zeros(1), uv, 0, False, 0.0, 2, None)
    fs = pg.FieldSet.from_spec(spec, storage="f32")
    lon = rng.uniform(lon_ax[20], lon_ax[-20], 30_000).astype(np.float32)
    lat = rng.uniform(-0.02, 0.02, 30_000).astype(np.float32)
    out, at_face = [], 0
    for chunk in (0, 5):
        ps = pg.ParticleSet(fs, lon, lat, pos="f32")
        ps.set_tune(block=128, resort_steps=0, chunk_steps=chunk)
        ps.execute(pg.Kernel("rk4"), 100 * 2.0, 2.0)
        out.append(ps.get())
    at_face = ((out[0]["lon"] - lon_ax[0]) % 41.0 == 0).sum()
    assert at_face > 100 and (out[0]["status"] == 0).mean() > 0.9
    _same(out[0], out[1])


def test_settled_on_a_level_from_above(pg):
    """Particles that sink onto a level and stay there (the settle behaviour
    reaches the dwelling depth exactly), 47 m below the level above it."""
    rng = np.random.default_rng(5)
    nx, ny = 24, 13
    spec = synth.FieldSpec(np.arange(nx) * 15.0, -45.0 + 7.5 * np.arange(ny),
                           np.array([0.0, 47.0, 94.0]), np.zeros(1),
                           rng.normal(size=(1, 2, 3, ny, nx)) * 3.0, 1, True, 0.0, 2, None)
    fs = pg.FieldSet.from_spec(spec, storage="f32")
    fs.add_constant("w_sink", 40.0 / H)
    fs.add_constant("dwelling_depth", 47.0)
    lon = rng.uniform(0.0, 360.0, 20_000).astype(np.float32)
    lat = rng.uniform(-30.0, 30.0, 20_000).astype(np.float32)
    dep = np.full(20_000, 20.0, np.float32)
    out = []
    for chunk in (0, 9):
        ps = pg.ParticleSet(fs, lon, lat, dep, pos="f32")
        ps.set_tune(block=128, resort_steps=0, chunk_steps=chunk)
        ps.execute(pg.Kernel("rk4", ("settle",), w_sink=None), 100 * 1800.0, 1800.0)
        out.append(ps.get())
    assert (out[0]["depth"] == 47.0).mean() > 0.9
    _same(out[0], out[1])


@pytest.mark.parametrize("nz", [1, 3])
def test_particles_on_the_last_nodes_of_a_closed_domain(pg, nz):
    """Flow along the walls of a flat box (no velocity across them): particles on
    the last node of an axis belong to the last cell and move as in the FP64 form."""
    rng = np.random.default_rng(6)
    nx, ny = 21, 17
    lon_ax, lat_ax = 41.0 * np.arange(nx), -8.0 * 47.0 + 47.0 * np.arange(ny)
    dep_ax = np.array([0.0, 20.0, 61.0]) if nz > 1 else np.zeros(1)
    nf = 3 if nz > 1 else 2
    v = rng.normal(size=(1, nf, nz, ny, nx)).astype(np.float32).astype(np.float64) * 0.25
    v[:, 0, :, :, [0, -1]] = 0.0
    v[:, 1, :, [0, -1], :] = 0.0
    if nz > 1:
        v[:, 2, [0, -1]] = 0.0
    spec = synth.FieldSpec(lon_ax, lat_ax, dep_ax, np.zeros(1), v, 0, False, 0.0, nf, None)
    n = 3000
    p = [rng.uniform(a[0] + 1.0, a[-1] - 1.0, n) if len(a) > 1 else np.zeros(n)
         for a in (lon_ax, lat_ax, dep_ax)]
    p[0][:1000] = lon_ax[-1]
    p[1][500:1500] = lat_ax[-1]
    p[2][1200:2200] = dep_ax[-1]
    p = [q.astype(np.float32).astype(np.float64) for q in p]
    out = []
    for pos, storage in (("f32", "f32"), ("f64", "f64")):
        fs = pg.FieldSet.from_spec(spec, storage=storage)
        ps = pg.ParticleSet(fs, p[0], p[1], p[2] if nz > 1 else None, pos=pos)
        ps.execute(pg.Kernel("rk4"), 100.0, 10.0)
        out.append(ps.get())
    a, b = out
    # rounding may put an FP32 result just outside where FP64's stays inside
    assert (b["status"] == 0).mean() > 0.9 and (a["status"] != b["status"]).mean() < 0.01
    both = (a["status"] == 0) & (b["status"] == 0)
    e = cell_error(a, b, spec, periodic=False)[both]
    assert np.mean(e) < 1e-3 and np.max(e) < 2e-2, (np.mean(e), np.max(e))
    for k, (ax, lo, hi) in dict(lon=(lon_ax, 0, 1000), lat=(lat_ax, 500, 1500)).items():
        assert (a[k][lo:hi] == ax[-1]).all()
