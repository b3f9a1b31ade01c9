"""pm_deposit_shape: column lengths that differ, and contexts without a choice."""
import numpy as np
import pytest

from test_deposit_gpu import load
from test_parity_gpu import pm, rel  # noqa: F401  (pm is a fixture)

pytestmark = pytest.mark.gpu


# 64 and 72 vertices along z in columns of 11 and 12 (FP64) or 6 (FP32) and half of it: of several lengths, with remainders
@pytest.mark.parametrize("n", [64, 72])
@pytest.mark.parametrize("precision,bound", [("PM_FP64", 1e-12), ("PM_MIXED", 2e-6)])
def test_column_lengths_agree(pm, n, precision, bound):  # noqa: F811
    """The same sums but for the order of additions: FP64 to 1e-12 and FP32 to 2e-6 of a field's norm."""
    pos = load("dense", n, n)
    mom = np.random.default_rng(n).standard_normal(pos.shape) * 1e-3
    runs = []
    for shape in (0, 1):
        g = pm.PM(n, len(pos), 10.0 * n, 0.31, 20.0, 0.0, 100, getattr(pm, precision))
        g.set_particles(pos, mom)
        assert pm.pm_deposit_shape(g.ctx, shape) == shape
        g.project()
        runs.append([g.field(f) for f in ("R", "Fx", "Fz", "Sxx", "Syz")])
        g.close()
    assert all(rel(b, a) < bound for a, b in zip(*runs))


def test_mixed_newtonian_has_no_choice(pm):  # noqa: F811
    """Timing launches nothing and keeps shape 0; a forced shape is kept and reported, as it was."""
    pos = np.random.default_rng(3).random((4096, 3))
    g = pm.PM(16, len(pos), 100.0, 0.31, 20.0, 0.0, 100, pm.PM_MIXED, pm.PM_NEWTONIAN)
    g.set_particles(pos, np.zeros_like(pos))
    g.step()
    assert pm.pm_deposit_shape(g.ctx, 1) == 1 and pm.pm_deposit_shape(g.ctx, -2) == 1
    g.timings()
    assert pm.pm_deposit_shape(g.ctx, -1) == 0
    assert g.timings()[1] == 0
    g.close()
