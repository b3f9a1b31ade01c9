"""FP64 drift: which cell a particle lands in, at the edges of the rule that finds it."""
import numpy as np
import pytest

from test_parity_gpu import make_pair, pm  # noqa: F401  (pm is a fixture)

pytestmark = pytest.mark.gpu

N = 16


def lattice():
    i = np.arange(N) / N
    return np.stack(np.meshgrid(i, i, i, indexing="ij"), -1).reshape(-1, 3)


@pytest.mark.parametrize("newtonian", [False, True])
@pytest.mark.parametrize("u", [0.0, 1e-20, -1e-20])
def test_offset_that_rounds_to_one(pm, newtonian, u):  # noqa: F811
    """On cell edges of a uniform load nothing moves by more than rounding: the force vanishes."""
    pos = lattice()
    _, g, *_ = make_pair(pm, N, 0, 10.0 * N, 1, pm.PM_FP64, newtonian=newtonian, zi=9.0, nsteps=20, pos=pos,
                         mom=np.full_like(pos, u))
    g.step()
    x, _ = g.particles()
    g.close()
    assert (x >= 0).all() and (x < 1).all()
    d = np.abs(x - pos)
    assert np.minimum(d, 1 - d).max() < 1e-13


@pytest.mark.parametrize("u", [1e9, -1e9, 1e12, -1e12, 1e17, -1e17, 1e300, -1e300])
def test_move_of_n_cells_keeps_the_cell(pm, u):  # noqa: F811
    """A Newtonian momentum that would carry a particle over N cells or more leaves it in its cell."""
    pos = lattice()
    mom = np.zeros_like(pos)
    mom[::5, 0] = u
    mom[1::5, 2] = u
    _, g, *_ = make_pair(pm, N, 0, 10.0 * N, 1, pm.PM_FP64, newtonian=True, zi=9.0, nsteps=20, pos=pos, mom=mom)
    g.step()
    x, _ = g.particles()
    g.close()
    moved = mom != 0
    cell = np.rint(pos * N)
    off = x * N - cell
    assert (off[moved] >= 0).all() and (off[moved] <= 1).all()
    d = np.abs(x - pos)[~moved]
    assert np.minimum(d, 1 - d).max() < 1e-13
