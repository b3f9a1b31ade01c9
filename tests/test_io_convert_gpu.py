"""f64 particle rows to cell + offset records and back: the integer-pipe conversions against IEEE arithmetic."""
import numpy as np
import pytest

from test_parity_gpu import pm  # noqa: F401  (a fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [8, 24, 72, 192, 256])
def test_load_and_store_round_as_ieee(pm, n):  # noqa: F811
    """Bit for bit: cell floor(x N), offset and momentum rounded to FP32, (cell + offset) / N back in FP64."""
    rng = np.random.default_rng(n)
    x = rng.random((4096, 3))
    k = rng.integers(0, n, 3000)
    x.reshape(-1)[:3000] = (k + rng.choice([0.0, 2.0 ** -24, 2.0 ** -25, 2.0 ** -45, 1 - 2.0 ** -24, 1 - 2.0 ** -26,
                                            0.5, 3e-39 * n], 3000)) / n
    x.reshape(-1)[3000:3012] = [0.0, -0.0, 1.0, -1.0, 1 - 2.0 ** -53, -2.0 ** -60, 5e-324, 1e-310, 2.25, -0.75, 7.0, 1e9]
    u = rng.standard_normal(x.shape) * 10.0 ** rng.integers(-12, 3, x.shape)
    u.reshape(-1)[:8] = [0.0, -0.0, 1e-40, -1e-45, 1e-60, 1.17549435e-38, 3.4e38, -2.0 ** -149]
    with np.errstate(under="ignore"):
        y = x - np.floor(x)
        y[y >= 1.0] = 0.0
        s = y * n
        c = np.floor(s).astype(np.int64)
        f = (s - np.floor(s))
        c[c >= n] -= n
        f32 = f.astype(np.float32)
        up = f32 >= 1
        f32[up] = 0
        c[up] = (c[up] + 1) % n
        u32 = u.astype(np.float32)
    g = pm.PM(n, len(x), 100.0, 0.31, 10.0, 0.0, 10, pm.PM_MIXED)
    g.set_particles(x, u)
    rec = np.zeros(len(x), pm.PACKED)
    pm.pm_get_particles_packed(g.ctx, len(x), rec)
    pos, mom = g.particles()
    g.close()
    assert np.array_equal(rec["cell"], (c[:, 2] * n + c[:, 1]) * n + c[:, 0])
    assert np.array_equal(rec["f"].view(np.uint32), f32.view(np.uint32))
    assert np.array_equal(rec["u"].view(np.uint32), u32.view(np.uint32))
    assert np.array_equal(pos, (c + f32.astype(np.float64)) * (1.0 / n))
    assert np.array_equal(mom.view(np.uint64), u32.astype(np.float64).view(np.uint64))
    d = pm.PM(n, len(x), 100.0, 0.31, 10.0, 0.0, 10, pm.PM_FP64)
    d.set_particles(x, u)
    pos, mom = d.particles()
    d.close()
    c = np.floor(s).astype(np.int64)
    c[c >= n] -= n
    assert np.array_equal(pos, (c + f) * (1.0 / n)) and np.array_equal(mom, u)
