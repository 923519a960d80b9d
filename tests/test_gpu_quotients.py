"""The FP64 form's quotients -- a position's fraction of its cell on each axis
and a time's fraction of its snapshot interval (Sect. 2.3, 2.4) -- are the
divisions' values, rounded to nearest, also where the exact quotient lies as
close as two doubles allow to the middle between two others (relative
distance 2^-107)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pg():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    import paper_1707_05163_gb300 as pg
    pg.load()
    return pg


def _next_to_middles(d):
    """Whole numbers a < d of 53 bits with 2^54 a = d M + e for an odd M of 54
    bits (the middle between two 53-bit quotients is M 2^-54) and e = 1 or -1."""
    out = []
    for e in (1, -1):
        m = -e * pow(d, -1, 1 << 54) % (1 << 54)
        a = (d * m + e) >> 54
        if m >> 53 and 1 << 52 <= a < d - (1 << 40):
            out.append(a)
    return out


def _pairs():
    rng = np.random.default_rng(7)
    divisors = [8116680080321247, (1 << 53) - 1, (1 << 53) - 3]
    divisors += [int(v) | 1 for v in rng.integers((1 << 52) + (1 << 50), 1 << 53, 60)]
    return [(a, d) for d in divisors for a in _next_to_middles(d)]


@pytest.mark.parametrize("axis", ["lon", "lat", "depth", "time"])
def test_fractions_next_to_a_rounding_middle_are_the_divisions(pg, axis):
    """One Euler step of one second from position 0 in a field whose velocity
    is the fraction itself: the new position is the fraction."""
    pairs = _pairs()
    assert len(pairs) > 16 and (7639898285114099, 8116680080321247) in pairs
    got, want = [], []
    for a, d in pairs:
        start, width = a * 2.0 ** -33, d * 2.0 ** -33     # about a million
        ax = {k: np.array([0.0, 2.0]) for k in ("lon", "lat")}
        if axis != "time":
            ax[axis] = np.array([0.0, width])
        fs = pg.FieldSet(ax["lon"], ax["lat"], ax.get("depth"), mesh="flat", nfields=2, storage="f64")
        times = np.array([0.0, width]) if axis == "time" else np.zeros(1)
        fs.set_times(times)
        for s in range(len(times)):
            v = np.zeros((2, 2 if axis == "depth" else 1, 2, 2))
            if axis == "lon":
                v[1, :, :, 1] = 1.0
            elif axis == "lat":
                v[0, :, 1, :] = 1.0
            elif axis == "depth":
                v[1, 1] = 1.0
            else:
                v[1] = float(s)
            fs.load_snapshot(s, v)
        p = {k: np.array([start if k == axis else 0.0]) for k in ("lon", "lat", "depth")}
        ps = pg.ParticleSet(fs, p["lon"], p["lat"], p["depth"], t0=start if axis == "time" else 0.0,
                            pos="f64")
        ps.execute(pg.Kernel("euler"), 1.0, 1.0)
        g = ps.get()
        assert g["status"][0] == 0 and g["step"][0] == 1
        got.append(g["lon" if axis == "lat" else "lat"][0])
        want.append(float(a) / float(d))
    np.testing.assert_array_equal(got, want)
