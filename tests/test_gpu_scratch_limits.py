"""Making and reading back a set needs little device memory beside its own
arrays: where a staging buffer for all positions does not fit, host positions go
through a smaller one piece by piece, with the same results; FP64 positions need
none.  The library's allocation limit (a host-side hook) stands in for a full
device."""
import numpy as np
import pytest

import synth
from tests.helpers import DAY

pytestmark = pytest.mark.gpu

N = 300_001
STAGE = 1_000_000                 # bytes: seven pieces or more


@pytest.fixture(scope="module")
def pg():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    import paper_1707_05163_gb300 as pg
    pg.load()
    return pg


class _Limit:
    def __init__(self, lib, extra):
        self.lib, self.extra = lib, extra

    def __enter__(self):
        assert self.lib.pg_debug_set_alloc_limit(self.extra) == 0

    def __exit__(self, *a):
        self.lib.pg_debug_set_alloc_limit(-1)


@pytest.mark.parametrize("with_depth", [True, False])
@pytest.mark.parametrize("pos,state,stage", [("f32", 49, STAGE), ("cell", 61, STAGE), ("f64", 61, 0)])
def test_sets_made_and_read_in_pieces(pg, pos, state, stage, with_depth):
    lib = pg.load()
    nx, ny, nz = 24, 13, 4
    rng = np.random.default_rng(1)
    spec = synth.FieldSpec(np.arange(nx) * 15.0, -45.0 + 7.5 * np.arange(ny), 10.0 * np.arange(nz),
                           np.zeros(1), rng.normal(size=(1, 2, nz, ny, nx)), 1, True, 0.0, 2, None)
    fs = pg.FieldSet.from_spec(spec, storage="f64" if pos == "f64" else "f32")
    lon = rng.uniform(-100.0, 460.0, N)
    lat = rng.uniform(-44.0, 44.0, N)
    dep = rng.uniform(0.0, 30.0, N) if with_depth else None
    time = np.where(np.arange(N) % 2, DAY, 0.0)
    whole = pg.ParticleSet(fs, lon, lat, dep, time=time, id_base=7, pos=pos)
    # the arrays (each on a 256-byte boundary), 16 bytes of counters, the staging
    with _Limit(lib, state * N + 12 * 256 + 16 + stage):
        ps = pg.ParticleSet(fs, lon, lat, dep, time=time, id_base=7, pos=pos)
    a, b = whole.get(), ps.get()
    for k in b:
        np.testing.assert_array_equal(a[k], b[k], err_msg=k)
    np.testing.assert_array_equal(b["id"], 7 + np.arange(N))
    np.testing.assert_array_equal(b["time"], time)
    np.testing.assert_array_equal(ps.get_variables()["age"], 0.0)
    with _Limit(lib, stage):
        c = ps.get()
    for k in c:
        np.testing.assert_array_equal(a[k], c[k], err_msg=k)
    # and no room at all: refused, unless nothing is staged
    if pos != "f64":
        with _Limit(lib, 0), pytest.raises(pg.PGError) as e:
            ps.get()
        assert e.value.code == -7
