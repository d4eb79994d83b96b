"""The energy on padded rows counts the grid's cells alone, whichever copy of
the state is the current one and whatever the device memory held before."""
import pytest

from parity_util import make_pair, params_kw

pytestmark = pytest.mark.gpu

TOL = 2e-5   # twice the bound on the fields: the energy is quadratic in them


@pytest.fixture
def used_memory():
    """Device memory that holds NaNs when it is handed out."""
    from paper_0809_1547_gb300.binding import mb_debug_fill_alloc
    mb_debug_fill_alloc(0xff)
    yield
    mb_debug_fill_alloc(-1)


# three padding cells and one; the many-steps launch of small grids and the
# single-pass step (tuned): an odd count, an even one, and past an adjoint
# call; no padding
@pytest.mark.parametrize("grid", [(49, 19, 22), (51, 22, 17), (139, 64, 33), (52, 17, 22)])
def test_energy_in_either_copy(grid, used_memory):
    from paper_0809_1547_gb300 import inputs
    eps, gain = inputs.random_small(grid, seed=3, npml=4, d_cells=4.0)
    o, g = make_pair(grid, eps, gain, 4e24, 1e13, 0x3E, params_kw(npml=4))
    src = ((grid[0] - 6, 9, 8), 2, 532e-9, 1.0e-15, 0.4e-15, 1e9)
    o.add_source(*src)
    g.set_source(*src)
    g.autotune()
    for n in (33, 1, 33):
        o.step(n)
        g.step(n)
        assert g.energy()[0] == pytest.approx(o.energy(), rel=TOL, abs=0)
    g.adjoint_energy_zface(5, 3)
    o.step(5)
    assert g.energy()[0] == pytest.approx(o.energy(), rel=TOL, abs=0)
    g.close()
