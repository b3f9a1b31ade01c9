"""Stage times of loads of another shape than one particle a cell, each against the same call on an even load.  The
bounds are ratios, far from what is measured on either side of the faults they stand for."""
import pytest

from test_parity_gpu import pm  # noqa: F401  (a fixture)

pytestmark = pytest.mark.gpu

N = 128


def make(pm, precision, flags, per_cell=1.0, clump=0):  # noqa: F811
    """An even (Poisson) load, a tenth of it in cells of `clump` particles."""
    import torch
    n = int(N ** 3 * per_cell)
    g = torch.Generator(device="cuda")
    g.manual_seed(11)
    pos = torch.rand((n, 3), generator=g, device="cuda", dtype=torch.float64)
    if clump:
        k = max(1, n // 10 // clump)
        c = torch.randint(0, N, (k, 3), generator=g, device="cuda").double().repeat_interleave(clump, 0)
        pos[:k * clump] = (c + pos[:k * clump]) / N
    s = pm.PM(N, n, 400.0, 0.31, 1.0, 0.0, 100, precision, flags)
    s.set_particles(pos, 1e-6 * torch.randn((n, 3), generator=g, device="cuda", dtype=torch.float64))
    return s


def power_ms(s):
    import torch
    s.power_spectrum(64)
    t = []
    for _ in range(5):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        s.power_spectrum(64)
        b.record()
        torch.cuda.synchronize()
        t.append(a.elapsed_time(b))
    return sorted(t)[2]


def test_fp64_power_of_clumps(pm):  # noqa: F811
    """A tenth of the mass in cells of 10^4: 1.3 times the even load (10 times in the deposit's columns)."""
    t = [power_ms(make(pm, pm.PM_FP64, pm.PM_NEWTONIAN, clump=c)) for c in (0, 10000)]
    assert t[1] < 3 * t[0], t
