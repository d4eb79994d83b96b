"""The default launch shapes of a context that was not tuned, on both sides of
the sizes where they change, give the bits of the plain walks."""
import numpy as np
import pytest

from parity_util import DT, DX

pytestmark = pytest.mark.gpu


# below and above 4, 6 and 8 M cells; rows of whole tiles of tensor copies and not
@pytest.mark.parametrize("grid", [(96, 90, 88), (160, 160, 155), (160, 160, 158), (192, 180, 176), (203, 200, 195),
                                  (203, 200, 200)])
def test_default_shapes(grid):
    from paper_0809_1547_gb300 import inputs
    from paper_0809_1547_gb300.binding import MBSimulation, mb_default_params
    eps, gain = inputs.random_small(grid, seed=4, npml=8, d_cells=12.0)
    sims = []
    for plain in (True, False):
        s = MBSimulation(grid, DX, DT, mb_default_params(npml=8))
        if plain:
            s.set_tuning((1, 32, 8, 16), (1, 32, 4, 16))
        s.set_step_launch((0, 0, 0, 0))
        s.set_material(eps, gain, 4e24, 1e13)
        s.set_seed(6)
        s.set_source(tuple(n // 2 for n in grid), 0, 532e-9, 1.0e-15, 0.4e-15, 1e9)
        s.step(30)
        sims.append(s)
    for f in ("Ex", "Ey", "Ez", "Hx", "Hz", "Px", "Jy", "N1", "N3"):
        np.testing.assert_array_equal(sims[1].field(f), sims[0].field(f), err_msg=f)
    for s in sims:
        s.close()
