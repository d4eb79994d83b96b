"""mb_get_field_device takes the destinations that a copy takes: any byte
address of the device, page-locked host memory."""
import ctypes

import numpy as np
import pytest

from parity_util import DT, DX

pytestmark = pytest.mark.gpu


# rows as they are (Ex: one copy) and padded; whole and ragged blocks of P
@pytest.mark.parametrize("grid", [(51, 13, 11), (52, 9, 7)])
@pytest.mark.parametrize("field", ["Ex", "Hz", "Px", "N3"])
def test_destinations(grid, field):
    import torch
    from paper_0809_1547_gb300.binding import FIELD_ID, MBSimulation, load_library, mb_default_params
    rng = np.random.default_rng(5)
    s = MBSimulation(grid, DX, DT, mb_default_params(npml=2))
    eps = np.where(rng.random(s.shape) < 0.5, 8.41, 1.0).astype(np.float32)
    s.set_material(eps, (eps < 2.0).astype(np.uint8), 4e24, 1e13)
    s.set_field(field, rng.standard_normal(s.shape).astype(np.float32))
    want = s.field_device(field)[0].cpu().numpy().reshape(-1)
    n = want.size
    dev = torch.zeros(4 * n + 16, dtype=torch.uint8, device="cuda")
    host = torch.zeros(n, dtype=torch.float32).pin_memory()
    torch.cuda.synchronize()
    for off in (0, 4, 1, 2, 7):
        rc = load_library().mb_get_field_device(s._h, FIELD_ID[field], ctypes.c_void_p(dev.data_ptr() + off), None)
        assert rc == 0, off
        got = dev.cpu().numpy()[off:off + 4 * n].copy().view(np.float32)
        np.testing.assert_array_equal(got, want, err_msg=str(off))
    rc = load_library().mb_get_field_device(s._h, FIELD_ID[field], ctypes.c_void_p(host.data_ptr()), None)
    assert rc == 0
    np.testing.assert_array_equal(host.numpy(), want)
    s.close()
