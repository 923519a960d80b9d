"""Particles added to a set between re-sorts (a daily release, Sect. 3): ages,
RKF45 step lengths and everything that depends on them are those of a set that
was made whole and never re-sorted.

A re-sort leaves ages and step lengths that no kernel has used where they are
and swaps the set's two copies of its arrays, so each entry of either copy has
to hold a new particle's zero -- also the entries that only a later ``add``
within the grown capacity fills."""
import numpy as np
import pytest

import synth
from tests.helpers import DAY

pytestmark = pytest.mark.gpu

N0, N1, N2 = 40_000, 4_000, 8_000      # capacity 60,000 after the first add


@pytest.fixture(scope="module")
def pg():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    import paper_1707_05163_gb300 as pg
    pg.load()
    return pg


def _fieldset(pg, pos):
    gf = synth.GlobalField(res_deg=4.0, nz=1, nt=3, seed=5, kmax=10, period=3 * DAY)
    fs = pg.FieldSet.from_spec(gf.spec(materialise=True), storage="f64" if pos == "f64" else "f32")
    fs.add_constant("max_age", 1.25 * DAY)
    fs.add_constant("rkf45_tol", 50.0)
    fs.add_constant("rkf45_min_dt", 60.0)
    fs.add_constant("rkf45_max_dt", 7200.0)
    return fs


def _ages_and_steps(ps, path, pos):
    """Ages, and the step lengths of a saved checkpoint: a 48-byte header, then
    the state arrays one after another (positions, time, id, step, status,
    age, step length)."""
    ps.save(path)
    raw, n = open(path, "rb").read(), len(ps)
    el = 8 if pos == "f64" else 4
    at = 48 + n * (3 * el + 8 + 8 + 4 + 1)
    age = np.frombuffer(raw, np.float64, n, at)
    hstep = np.frombuffer(raw, np.float64, n, at + 8 * n)
    assert len(raw) == at + 16 * n
    return age, hstep


@pytest.mark.parametrize("pos", ["f32", "f64"])
@pytest.mark.parametrize("then", ["age", "rkf45"])
def test_particles_added_between_resorts_start_from_zero(pg, tmp_path, pos, then):
    fs = _fieldset(pg, pos)
    n = N0 + N1 + N2
    lon, lat, _ = synth.uniform_particles(n, 9, (0, 360), (-60, 60), dtype=np.float32)
    # earlier sets of the same size leave other values in the memory they free
    for _ in range(2):
        old = pg.ParticleSet(fs, np.resize(lon, 60_000), np.resize(lat, 60_000), pos=pos)
        old.set_tune(0, 10, 0)
        old.execute(pg.Kernel("rkf45", ("age",)), 0.5 * DAY, 3600.0)
        old.destroy()
    ps = pg.ParticleSet(fs, lon[:N0], lat[:N0], pos=pos)
    ps.add(lon[N0:N0 + N1], lat[N0:N0 + N1], id_base=N0)        # grows: 60,000 entries
    ps.resort()
    ps.add(lon[N0 + N1:], lat[N0 + N1:], id_base=N0 + N1)       # within the capacity
    ps.resort()
    assert len(ps) == n
    age, hstep = _ages_and_steps(ps, tmp_path / "set.bin", pos)
    np.testing.assert_array_equal(age, 0.0)
    np.testing.assert_array_equal(hstep, 0.0)
    # and the runs that start from them
    kernel = pg.Kernel("rk4", ("age",)) if then == "age" else pg.Kernel("rkf45")
    ref = pg.ParticleSet(fs, lon, lat, pos=pos)
    for s in (ps, ref):
        s.set_tune(0, 0, 24)
        s.execute(kernel, 1.5 * DAY, 3600.0)
    a, b = ps.get(), ref.get()
    for k in ("id", "lon", "lat", "time", "step", "status"):
        np.testing.assert_array_equal(a[k], b[k], err_msg=k)
    if then == "age":
        assert (b["status"] == 4).mean() > 0.9
