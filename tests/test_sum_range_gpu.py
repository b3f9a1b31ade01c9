"""The T00 sums and the density contrast of mixed contexts where one vertex holds very many particles, or particles of
very unequal charge."""
import numpy as np
import pytest

from test_parity_gpu import pm  # noqa: F401  (a fixture)
from test_power_gpu import reference

pytestmark = pytest.mark.gpu

CROWD = 300000


def load(n, seed):
    """n^3 spread particles and CROWD in one cell, with offsets that FP32 holds."""
    rng = np.random.default_rng(seed)
    cell = np.concatenate([rng.integers(0, n, (n ** 3, 3)), np.full((CROWD, 3), 5)])
    f = rng.integers(0, 1 << 24, cell.shape) / 2.0 ** 24
    return (cell + f) / n


def source(pm, n, pos, mom, precision):  # noqa: F811
    g = pm.PM(n, len(pos), 160.0, 0.31, 20.0, 0.0, 100, precision)
    g.set_particles(pos, mom)
    g.project()
    r = g.field("R")
    g.close()
    return r


# crowded: 37500 charges a vertex, a mean of 2; fast: E = 1e4 a
@pytest.mark.parametrize("kind,n", [("crowded", 64), ("fast", 16)])
def test_mixed_source_of_a_crowded_vertex(pm, kind, n):  # noqa: F811
    """R against an FP64 context with the same particles, to 5e-7 of its largest value: a term has five roundings of
    2^-24 at most (weights, charge, product) that lean one way only where they are the same for all (mass, a: two), and
    the sums add none.  A plain FP32 sum of 3e5 terms is 3e5^(1/2) roundings off, 3e-5."""
    pos = load(n, 3)
    mom = np.random.default_rng(4).standard_normal(pos.shape)
    mom *= (1e4 / 21 if kind == "fast" else 1e-5) / np.linalg.norm(mom, axis=1)[:, None]
    mom = mom.astype(np.float32).astype(np.float64)
    a, b = (source(pm, n, pos, mom, p) for p in (pm.PM_FP64, pm.PM_MIXED))
    assert abs(b - a).max() < 5e-7 * abs(a).max()


def test_mixed_power_of_a_crowded_vertex(pm):  # noqa: F811
    """P(k) of a contrast that is one spike of 8 vertices, in the bins where its spectrum is flat.  The transform of a
    spike takes log2 N^3 = 18 additions with one term each that is not small, so a mode is within 18 roundings of 2^-24,
    its square within 2.2e-6; the contrast itself is exact to FP32 (a plain FP32 sum of 3e5 terms is 1e-5 off)."""
    n = 64
    pos = load(n, 7)
    g = pm.PM(n, len(pos), 100.0, 0.31, 10.0, 0.0, 10, pm.PM_MIXED, pm.PM_NEWTONIAN)
    g.set_particles(pos, np.zeros_like(pos))
    k, pk, nm = g.power_spectrum(n // 4)
    g.close()
    rk, rp, rn = reference(n, pos, n // 4)
    assert np.array_equal(nm, rn) and np.allclose(pk, rp, rtol=2.2e-6, atol=0)
