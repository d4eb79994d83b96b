"""P, J and the populations sit in blocks of eight cells on the device: every
way in and out (host and device reads, writes, saved states) speaks the grid's
own order, on grids whose cells or rows do not fill whole blocks, before and
after a material is set."""
import numpy as np
import pytest

from parity_util import DT, DX

pytestmark = pytest.mark.gpu

GAIN = ("Px", "Py", "Pz", "Jx", "Jy", "Jz", "N1", "N2", "N3")
FIELDS = ("Ex", "Ey", "Ez", "Hx", "Hy", "Hz") + GAIN


# rows, planes and the whole grid off the block length; one cell short of and
# past whole blocks; padded rows
@pytest.mark.parametrize("grid", [(17, 5, 3), (5, 3, 1), (8, 3, 3), (51, 13, 11), (64, 9, 7)])
@pytest.mark.parametrize("material", [False, True])
def test_every_field_in_and_out(grid, material):
    from paper_0809_1547_gb300.binding import MBSimulation, mb_default_params
    s = MBSimulation(grid, DX, DT, mb_default_params(npml=0))
    rng = np.random.default_rng(5)
    if material:
        eps = np.where(rng.random(s.shape) < 0.5, 8.41, 1.0).astype(np.float32)
        s.set_material(eps, (eps < 2.0).astype(np.uint8), 4e24, 1e13)
    names = FIELDS if material else [f for f in FIELDS if f[0] != "N"]
    want = {f: rng.standard_normal(s.shape).astype(np.float32) for f in names}
    for f in names:
        s.set_field(f, want[f])
    for f in names:
        np.testing.assert_allclose(s.field(f), want[f], rtol=1e-6, err_msg=f)
        t, scale = s.field_device(f)
        np.testing.assert_allclose(t.cpu().numpy() * scale, want[f], rtol=1e-5, err_msg=f)
    blob = s.save_state()
    n = int(np.prod(grid))
    at = np.frombuffer(blob, np.float32, 15 * n, offset=32).reshape((15,) + s.shape)
    for q, f in enumerate(FIELDS):   # the blob's order
        if f in names:
            np.testing.assert_allclose(at[q] * np.float32(s.field_device(f)[1]), want[f], rtol=1e-5, err_msg=f)
    for f in names:
        s.set_field(f, np.zeros(s.shape, np.float32))
    s.load_state(blob)
    for f in names:
        np.testing.assert_allclose(s.field(f), want[f], rtol=1e-6, err_msg=f)
    if material:   # a new material clears them
        s.set_material(eps, (eps < 2.0).astype(np.uint8), 4e24, 1e13)
        for f in GAIN:
            assert not s.field(f).any(), f
    s.close()
