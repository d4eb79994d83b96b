"""Fields and states are read and written where the device has no memory left
for the packed copy that padded rows and the blocks of P, J and n go through."""
import numpy as np
import pytest

from parity_util import DT, DX

pytestmark = pytest.mark.gpu

FIELDS = ("Ex", "Ey", "Ez", "Hx", "Hy", "Hz", "Px", "Py", "Pz", "Jx", "Jy", "Jz")


@pytest.mark.parametrize("grid", [(51, 13, 11), (52, 9, 7)])
def test_fields_without_device_memory(grid):
    from paper_0809_1547_gb300.binding import MBSimulation, mb_debug_fail_alloc, mb_default_params
    rng = np.random.default_rng(5)
    want = {f: rng.standard_normal(grid[::-1]).astype(np.float32) for f in FIELDS}
    a, b = (MBSimulation(grid, DX, DT, mb_default_params(npml=2)) for _ in range(2))

    def refused(fn):   # without a material nothing is set aside for it yet
        mb_debug_fail_alloc(0)
        try:
            return fn()
        finally:
            mb_debug_fail_alloc(-1)
    for f in FIELDS:
        refused(lambda: a.set_field(f, want[f]))
        b.set_field(f, want[f])
    for f in FIELDS:
        np.testing.assert_array_equal(refused(lambda: a.field(f)), b.field(f), err_msg=f)
    blob = refused(a.save_state)
    assert bytes(blob) == bytes(b.save_state())
    c = MBSimulation(grid, DX, DT, mb_default_params(npml=2))
    refused(lambda: c.load_state(blob))
    for f in FIELDS:
        np.testing.assert_array_equal(c.field(f), b.field(f), err_msg=f)
    for s in (a, b, c):
        s.close()
