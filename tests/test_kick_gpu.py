"""Gather + kick + drift on loads that meet the edges of its tiles, against the FP64 oracle."""
import numpy as np
import pytest

from test_deposit_gpu import load
from test_parity_gpu import compare, make_pair, pm  # noqa: F401  (pm is a fixture)

pytestmark = pytest.mark.gpu


# rows of 24 and 32 cells, of 24 (48) and 24 (72) with several tiles along x; rows of more than 32 particles and none;
# momenta that carry particles over several cells and the box's edge (but not over N cells, where the step keeps the
# cell)
@pytest.mark.parametrize("n", [24, 32, 48, 72])
@pytest.mark.parametrize("kind", ["dense", "sparse", "edges"])
@pytest.mark.parametrize("newtonian", [False, True])
def test_fp64_kick_edges(pm, n, kind, newtonian):  # noqa: F811
    """1e-11, the bar of the whole step."""
    pos = load(kind, n, 11 * n)
    mom = np.random.default_rng(n).standard_normal(pos.shape) * 2e-2
    orc, g, *_ = make_pair(pm, n, 0, 10.0 * n, 1, pm.PM_FP64, newtonian=newtonian, zi=9.0, nsteps=20, pos=pos, mom=mom)
    for _ in range(3):
        orc.step()
        g.step()
    e = compare(orc, g, n, full=not newtonian)
    g.close()
    assert all(v < 1e-11 for v in e.values()), e
