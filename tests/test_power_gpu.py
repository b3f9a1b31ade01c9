"""The P(k) diagnostic against numpy in FP64: mesh sizes of every kind, empty and crowded cells, more and fewer bins
than the mesh has shells."""
import math

import numpy as np
import pytest

from test_deposit_gpu import load
from test_parity_gpu import pm  # noqa: F401  (a fixture)

pytestmark = pytest.mark.gpu


def reference(n, pos, nbins):
    s = pos * n
    c = np.floor(s).astype(np.int64)
    f = s - c
    rho = np.zeros(n ** 3)
    for i in range(8):
        d = np.array([i & 1, (i >> 1) & 1, i >> 2])
        w = np.where(d, f, 1 - f).prod(1)
        g = (c + d) % n
        np.add.at(rho, (g[:, 2] * n + g[:, 1]) * n + g[:, 0], w)
    dk = np.fft.rfftn((rho * (n ** 3 / len(pos)) - 1).reshape(n, n, n))
    a = np.fft.fftfreq(n, 1 / n)
    x = np.arange(n // 2 + 1)
    kn = np.sqrt(a[:, None, None] ** 2 + a[None, :, None] ** 2 + x[None, None, :] ** 2)
    wt = np.broadcast_to(np.where((x > 0) & (2 * x < n), 2.0, 1.0), kn.shape)
    b = np.rint(kn).astype(int).ravel()
    use = (b >= 1) & (b < nbins)
    tot = [np.bincount(b[use], (wt * q).ravel()[use], nbins) for q in (np.ones_like(kn), kn, np.abs(dk) ** 2 / n ** 6)]
    cnt = np.maximum(tot[0], 1)
    return 2 * math.pi * tot[1] / cnt, tot[2] / cnt, tot[0].astype(np.int64)


@pytest.mark.parametrize("n", [8, 24, 32, 72])
@pytest.mark.parametrize("kind", ["dense", "sparse"])
@pytest.mark.parametrize("mixed", [False, True])
def test_power_spectrum(pm, n, kind, mixed):  # noqa: F811
    """FP64 to 1e-12.  Mixed: offsets are FP32 here, so the contrast is exact to FP32 and the FP32 transform adds about
    5e-7 of the largest modes to each."""
    pos = load(kind, n, 3 * n)
    if mixed:   # offsets that FP32 holds
        s = pos * n
        pos = (np.floor(s) + (s - np.floor(s)).astype(np.float32).astype(np.float64).clip(0, 1 - 2.0 ** -24)) / n
    g = pm.PM(n, len(pos), 100.0, 0.31, 10.0, 0.0, 10, pm.PM_MIXED if mixed else pm.PM_FP64, pm.PM_NEWTONIAN)
    g.set_particles(pos, np.zeros_like(pos))
    for nbins in (2, n // 2 + 1, n + 3):
        k, pk, nm = g.power_spectrum(nbins)
        rk, rp, rn = reference(n, pos, nbins)
        assert np.array_equal(nm, rn) and np.allclose(k, rk, rtol=1e-12, atol=0)
        if mixed:
            assert np.allclose(pk, rp, rtol=2e-6, atol=1e-12 * rp.max())
        else:
            assert np.allclose(pk, rp, rtol=1e-12, atol=0)
    g.close()
