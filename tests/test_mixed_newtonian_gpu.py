"""The mixed Newtonian deposit and kick, with and without a force correction, on loads that meet the edges of their
tiles: cells and rows of very many particles, nearly empty ones, cell boundaries.  Against an FP64 context with the same
particles."""
import numpy as np
import pytest

from mixed_bounds import MIXED_BOUND
from test_deposit_gpu import load
from test_parity_gpu import pm, rel  # noqa: F401  (pm is a fixture)

pytestmark = pytest.mark.gpu


def particles(kind, n):
    pos = np.random.default_rng(n).random((16 * n ** 3, 3)) if kind == "full" else load(kind, n, 13 * n)
    c = np.floor(pos * n)
    pos = (c + (pos * n - c).astype(np.float32).clip(0, np.float32(1 - 2 ** -24))) / n
    mom = np.random.default_rng(n + 1).standard_normal(pos.shape) * 1e-3
    return pos, mom.astype(np.float32).astype(np.float64)


# rows of one tile (8, 24), of several with a remainder (72); dense: cells of 150 and 70 at the corner and beside each
# other; full: 16 a cell, tiles of a dozen chunks
@pytest.mark.parametrize("n,kind", [(8, "full"), (24, "full"), (24, "dense"), (72, "dense"), (24, "sparse"), (72, "sparse"),
                                    (72, "edges")])
@pytest.mark.parametrize("corrected", [False, True])
def test_mixed_newtonian_edges(pm, n, kind, corrected):  # noqa: F811
    """R to 1e-6 of its norm (a handful of roundings of 2^-24 a term, which the sums keep); momenta of two steps to the
    mixed bound; positions to 1e-5 of a cell: a drift below a cell, of which FP32 loses some 1e-7."""
    import torch
    pos, mom = particles(kind, n)
    corr = torch.zeros((n ** 3, 8), device="cuda")
    corr[:, :3] = 1e-4 * torch.randn((n ** 3, 3), generator=torch.Generator(device="cuda").manual_seed(n), device="cuda")
    got = {}
    for prec in (pm.PM_FP64, pm.PM_MIXED):
        g = pm.PM(n, len(pos), 10.0 * n, 0.31, 20.0, 0.0, 100, prec, pm.PM_NEWTONIAN)
        g.set_particles(pos, mom)
        if corrected:
            pm.pm_set_correction(g.ctx, corr)
        g.project()
        r = g.field("R")
        g.solve()
        g.update()
        g.step()
        got[prec] = (r, *g.particles())
        g.close()
    (r0, x0, u0), (r1, x1, u1) = got[pm.PM_FP64], got[pm.PM_MIXED]
    dx = (x1 - x0 + 0.5) % 1.0 - 0.5
    assert rel(r1, r0) < 1e-6 and rel(u1, u0) < MIXED_BOUND["u"] and np.abs(dx).max() * n < 1e-5
    assert np.linalg.norm(u0 - mom) > 1e-3 * np.linalg.norm(u0)   # the kick is not lost in the momenta
