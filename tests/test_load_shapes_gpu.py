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


def stage_ms(s, stage):
    for _ in range(2):
        s.step()
    s.timings()
    for _ in range(5):
        s.step()
    ms = s.timings()[0][stage]
    s.close()
    return ms


# a particle of a dense load (or of one with clumps) against one of an even load of one a cell
@pytest.mark.parametrize("precision,bound", [("PM_MIXED", 1.2), ("PM_FP64", 1.5)])
def test_deposit_of_a_dense_load(pm, precision, bound):  # noqa: F811
    """16 particles a cell cost 0.8 (FP32) and 0.6 (FP64) of the even load's time a particle; 1.5 and 2.3 where the
    vertex lanes sum them one by one."""
    t = [stage_ms(make(pm, getattr(pm, precision), 0, c), "project") / c for c in (1, 16)]
    assert t[1] < bound * t[0], t


@pytest.mark.parametrize("precision,bound", [("PM_MIXED", 3.0), ("PM_FP64", 2.0)])
def test_deposit_of_clumps(pm, precision, bound):  # noqa: F811
    """A tenth of the mass in cells of 1000: 2 (FP32) and 1.2 (FP64) times the even load; 4 and 3.3 before."""
    t = [stage_ms(make(pm, getattr(pm, precision), 0, 1.0, c), "project") for c in (0, 1000)]
    assert t[1] < bound * t[0], t


def test_fp64_kick_of_sparse_and_crowded_rows(pm):  # noqa: F811
    """0.05 particles a cell 0.3 and a tenth of the mass in cells of 1000 1.2 times the even load; 0.8 and 2 where each
    warp takes its own row."""
    t = [stage_ms(make(pm, pm.PM_FP64, 0, *load), "kick_drift") for load in ((1.0,), (0.05,), (1.0, 1000))]
    assert t[1] < 0.55 * t[0] and t[2] < 1.6 * t[0], t


def test_mass_deposit_of_a_dense_load(pm):  # noqa: F811
    """16 particles a cell cost 0.6 of the even load's time a particle in the mixed Newtonian deposit; 1.7 where a warp
    stages full cells one after another."""
    t = [stage_ms(make(pm, pm.PM_MIXED, pm.PM_NEWTONIAN, c), "project") / c for c in (1, 16)]
    assert t[1] < 1.1 * t[0], t


def test_mixed_kick_of_clumps(pm):  # noqa: F811
    """A tenth of the mass in cells of 1000: 1.3 times the even load; 2 where each warp takes its own row."""
    t = [stage_ms(make(pm, pm.PM_MIXED, 0, 1.0, c), "kick_drift") for c in (0, 1000)]
    assert t[1] < 1.6 * t[0], t


def test_mixed_clumps_move_as_in_fp64(pm):  # noqa: F811
    """Rows of far more than 96 particles beside ordinary ones, tiles with and without: every particle is moved once.
    Momenta of the mixed step to its bound, positions to 1e-5 of a cell (a drift far below a cell)."""
    import numpy as np
    from mixed_bounds import MIXED_BOUND
    from test_parity_gpu import rel
    rng = np.random.default_rng(17)
    n = 48
    cells = np.array([[0, 0, 0], [47, 47, 47], [23, 7, 8], [24, 8, 7], [10, 40, 16]])
    pos = np.concatenate([c + rng.integers(0, 1 << 24, (m, 3)) / 2.0 ** 24
                          for c, m in zip(cells, (400, 97, 96, 1000, 33))] +
                         [rng.integers(0, n, (n ** 3, 3)) + rng.integers(0, 1 << 24, (n ** 3, 3)) / 2.0 ** 24]) / n
    mom = (1e-3 * rng.standard_normal(pos.shape)).astype(np.float32).astype(np.float64)
    got = []
    for prec in (pm.PM_FP64, pm.PM_MIXED):
        g = pm.PM(n, len(pos), 10.0 * n, 0.31, 20.0, 0.0, 100, prec)
        g.set_particles(pos, mom)
        for _ in range(2):
            g.step()
        got.append(g.particles())
        g.close()
    (x0, u0), (x1, u1) = got
    assert rel(u1, u0) < MIXED_BOUND["u"] and np.abs((x1 - x0 + 0.5) % 1.0 - 0.5).max() * n < 1e-5
    assert np.abs(x1 - pos).max() > 0 and (u1 != mom).any(1).all()
