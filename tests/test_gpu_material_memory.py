"""A gain list that gets no memory leaves a context without a material, not one
whose lists are gone: it steps, and the next material is as on a new context."""
import numpy as np
import pytest

from parity_util import DT, DX

pytestmark = pytest.mark.gpu

STATE = ("Ex", "Ey", "Ez", "Hx", "Hy", "Hz", "Px", "Jz", "N1", "N2", "N3")


# padded rows (two lists) and rows as they are (one)
@pytest.mark.parametrize("grid,lists", [((51, 13, 11), 2), ((52, 13, 11), 1)])
def test_gain_list_without_memory(grid, lists):
    from paper_0809_1547_gb300.binding import (MB_ERR_OOM, MBError, MBSimulation, mb_debug_fail_alloc,
                                               mb_default_params)
    rng = np.random.default_rng(3)
    eps = np.where(rng.random(grid[::-1]) < 0.5, 8.41, 1.0).astype(np.float32)
    few, many = ((eps < 2.0) & (rng.random(eps.shape) < f) for f in (0.2, 0.9))

    def new():
        s = MBSimulation(grid, DX, DT, mb_default_params(npml=2))
        s.set_step_launch((0, 0, 0, 0))   # the passes that run over the list
        s.set_seed(8)
        s.set_source((25, 6, 5), 1, 532e-9, 1.0e-15, 0.4e-15, 1e9)
        return s
    for n in range(lists):
        a, b = new(), new()
        blob = a.save_state()
        a.set_material(eps, few.astype(np.uint8), 4e24, 1e13)
        a.step(4)
        mb_debug_fail_alloc(n)
        try:
            with pytest.raises(MBError) as e:
                a.set_material(eps, many.astype(np.uint8), 4e24, 1e13)
        finally:
            mb_debug_fail_alloc(-1)
        assert e.value.code == MB_ERR_OOM
        with pytest.raises(MBError):
            a.gain_list()
        a.load_state(blob)   # zero fields at step 0
        vacuum = new()
        for s in (a, vacuum):
            s.step(5)
        for f in ("Ex", "Ey", "Hz", "Px", "Jz"):
            np.testing.assert_array_equal(a.field(f), vacuum.field(f), err_msg=f)
        a.load_state(blob)
        for s in (a, b):   # fewer cells than the first list held
            s.set_material(eps, few.astype(np.uint8), 4e24, 1e13)
            s.step(9)
        for f in STATE:
            np.testing.assert_array_equal(a.field(f), b.field(f), err_msg=f)
        np.testing.assert_array_equal(a.gain_list(), b.gain_list())
        for s in (a, b, vacuum):
            s.close()
