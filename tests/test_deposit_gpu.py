"""The projection on loads that meet the edges of its tiles: every source field against the FP64 oracle."""
import numpy as np
import pytest

from test_parity_gpu import compare, make_pair, pm, rel  # noqa: F401  (pm is a fixture)

pytestmark = pytest.mark.gpu


def load(kind, n, seed):
    """Positions: `dense` fills a few cells with many particles (rows of far more than 32, cells at the periodic
    corner and beside it), `sparse` leaves most rows empty, `edges` puts particles on cell and box boundaries."""
    rng = np.random.default_rng(seed)
    if kind == "dense":
        cells = np.array([[0, 0, 0], [n - 1, n - 1, n - 1], [n - 1, 0, 0], [n // 2, 1, n - 1], [n // 2 - 1, 1, n - 1]])
        pos = np.concatenate([(c + rng.random((m, 3))) / n for c, m in zip(cells, (150, 70, 33, 32, 31))])
        return np.concatenate([pos, rng.random((2 * n * n, 3))])
    if kind == "sparse":
        return rng.random((n + 3, 3))
    pos = rng.integers(0, n, (4 * n * n, 3)) / n
    pos[::2] += (rng.random((len(pos[::2]), 3)) - 0.5) / n
    return pos % 1.0


# one tile (8), a closed row (24, 32), tiles of several rows and columns with remainders (48, 72)
@pytest.mark.parametrize("n", [8, 24, 32, 48, 72])
@pytest.mark.parametrize("kind", ["dense", "sparse", "edges"])
@pytest.mark.parametrize("newtonian", [False, True])
def test_fp64_projection_edges(pm, n, kind, newtonian):  # noqa: F811
    """FP64 sums of at most 2e3 terms a vertex: 1e-11, the bar of the whole step."""
    pos = load(kind, n, 7 * n)
    mom = np.random.default_rng(n).standard_normal(pos.shape) * 1e-3
    orc, g, *_ = make_pair(pm, n, 0, 10.0 * n, 1, pm.PM_FP64, newtonian=newtonian, zi=20.0, pos=pos, mom=mom)
    for _ in range(2):
        orc.step()
        g.step()
    e = compare(orc, g, n, full=not newtonian)
    r = rel(g.field("R"), orc.field("R"))
    g.close()
    assert all(v < 1e-11 for v in e.values()) and r < 1e-11, (e, r)


@pytest.mark.parametrize("n", [16, 32, 72])
@pytest.mark.parametrize("kind", ["dense", "sparse"])
def test_mixed_projection_edges(pm, n, kind):  # noqa: F811
    """FP32 charges and weights (2^-24 each, a handful of roundings a term) with the T00 sums in two words: R to
    1e-6 of its norm against the FP64 context of the same FP32-rounded particles, the FP32 sums to 2e-6."""
    pos = load(kind, n, 5 * n)
    pos = (np.floor(pos * n) + np.float32(pos * n - np.floor(pos * n)).clip(0, np.float32(1 - 2 ** -24))) / n
    mom = (np.random.default_rng(n).standard_normal(pos.shape) * 1e-3).astype(np.float32).astype(np.float64)
    got = {}
    for prec in (pm.PM_FP64, pm.PM_MIXED):
        g = pm.PM(n, len(pos), 10.0 * n, 0.31, 20.0, 0.0, 100, prec)
        g.set_particles(pos, mom)
        g.project()
        got[prec] = {f: g.field(f) for f in ("R", "Fx", "Fz", "Sxx", "Syz")}
        g.close()
    off = {f: rel(got[pm.PM_MIXED][f], got[pm.PM_FP64][f]) for f in got[pm.PM_FP64]}
    assert off["R"] < 1e-6 and all(v < 2e-6 for v in off.values()), off
