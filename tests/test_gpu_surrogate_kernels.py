"""A surrogate run whose checking kernel has ages or adaptive steps: the run's own
particle sets start them from zero, whatever the memory they get held before.
With a threshold of zero every particle takes the checking kernel's state, which
over one block is that of the kernel by itself."""
import numpy as np
import pytest

import synth
from tests.helpers import DAY

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pg():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    import paper_1707_05163_gb300 as pg
    pg.load()
    return pg


@pytest.mark.parametrize("n", [1, 4000])
@pytest.mark.parametrize("scheme,behaviours", [("rkf45", ()), ("rk4", ("age",))])
def test_a_checked_block_is_the_checking_kernels_own_run(pg, n, scheme, behaviours):
    gf = synth.GlobalField(res_deg=2.0, nz=8, nt=6, seed=41, kmax=20, period=6 * DAY)
    fs = pg.FieldSet.from_spec(gf.spec(materialise=True), storage="f32")
    fs.add_constant("max_age", 1.5 * DAY)
    fs.add_constant("rkf45_tol", 10.0)
    fs.add_constant("rkf45_min_dt", 60.0)
    fs.add_constant("rkf45_max_dt", 7200.0)
    lon, lat, dep = synth.uniform_particles(n, 12, (0, 360), (-60, 60), (10.0, 800.0),
                                            dtype=np.float32)
    for _ in range(3):          # sets of the same size leave ages and step lengths behind
        old = pg.ParticleSet(fs, lon, lat, dep, pos="f32")
        old.execute(pg.Kernel("rkf45", ("age",)), DAY, 1800.0)
        old.destroy()
    kernel = pg.Kernel(scheme, behaviours)
    ref = pg.ParticleSet(fs, lon, lat, dep, pos="f32")
    ref.execute(kernel, DAY, 1800.0)
    ps = pg.ParticleSet(fs, lon, lat, dep, pos="f32")
    net = pg.MLP(37, 256, 4, 3, seed=3)
    pg.surrogate_run(ps, net, kernel, nsteps=1, check_every=1, threshold=0.0)
    a, b = ps.get(), ref.get()
    assert (b["status"] == 0).mean() > 0.9
    for k in ("lon", "lat", "depth", "time", "status"):
        np.testing.assert_array_equal(a[k], b[k], err_msg=k)
