"""The FFT passes of every kind of mesh size: the Poisson solve of a random source against FFTs of torch in FP64."""
import math

import numpy as np
import pytest

from test_parity_gpu import pm  # noqa: F401  (a fixture)

pytestmark = pytest.mark.gpu


def solve_error(pm, n, precision):  # noqa: F811
    import torch
    rng = np.random.default_rng(n)
    pos = rng.random((20000, 3))
    g = pm.PM(n, len(pos), 300.0, 0.31, 20.0, 0.0, 100, precision, pm.PM_NEWTONIAN)
    g.set_particles(pos, np.zeros_like(pos))
    g.project()
    r = torch.empty((n, n, n), dtype=torch.float64, device="cuda")
    phi = torch.empty_like(r)
    pm.pm_get_field(g.ctx, "R", r)
    g.solve()
    pm.pm_get_field(g.ctx, "phi", phi)
    torch.cuda.synchronize()
    g.close()
    k = 2 * n * torch.sin(math.pi * torch.fft.fftfreq(n, device="cuda", dtype=torch.float64))
    kx = 2 * n * torch.sin(math.pi * torch.fft.rfftfreq(n, device="cuda", dtype=torch.float64))
    k2 = k[:, None, None] ** 2 + k[None, :, None] ** 2 + kx[None, None, :] ** 2
    rk = torch.fft.rfftn(r)
    rk[0, 0, 0] = 0
    k2[0, 0, 0] = 1
    want = torch.fft.irfftn(-rk / k2, s=(n, n, n))
    return float((phi - want).norm() / want.norm())


@pytest.mark.parametrize("n", [8, 24, 72, 144, 216, 288, 432, 648, 864])
def test_mixed_sizes(pm, n):  # noqa: F811
    """FP32 transforms: about sqrt(log2 N^3) roundings of 2^-24 each way, below 5e-7."""
    assert solve_error(pm, n, pm.PM_MIXED) < 5e-7


@pytest.mark.parametrize("n", [8, 24, 72, 96, 144, 216, 288])
def test_fp64_sizes(pm, n):  # noqa: F811
    assert solve_error(pm, n, pm.PM_FP64) < 1e-14
