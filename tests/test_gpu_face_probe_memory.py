"""Face probes whose device memory cannot be had are off, not half there."""
import numpy as np
import pytest

from parity_util import DT, DX

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("launch", [(0, 0, 0, 0), (1, 32, 4, 4)])
@pytest.mark.parametrize("failing", [0, 1, 2, 3])   # frequencies, FP64 sums, FP32 sums, read-out sums
def test_no_memory_for_face_probes(failing, launch):
    from paper_0809_1547_gb300.binding import (MB_ERR_OOM, MB_ERR_STATE, MBError, MBSimulation,
                                               mb_debug_fail_alloc, mb_default_params)
    sims = []
    for _ in range(2):
        s = MBSimulation((32, 20, 18), DX, DT, mb_default_params(npml=4))
        s.set_step_launch(launch)
        s.set_source((16, 10, 9), 2, 532e-9, 1.0e-15, 0.4e-15, 1e9)
        s.add_face_probes(2, 2, 8, 500e-9, 650e-9)
        s.step(4)   # graphs that hold the first sums
        sims.append(s)
    a, b = sims
    mb_debug_fail_alloc(failing)
    try:
        with pytest.raises(MBError) as e:
            a.add_face_probes(3, 2, 8, 500e-9, 650e-9)
    finally:
        mb_debug_fail_alloc(-1)
    assert e.value.code == MB_ERR_OOM
    with pytest.raises(MBError) as e:
        a.face_spectrum(0)
    assert e.value.code == MB_ERR_STATE
    for s in sims:
        s.step(6)
        s.add_face_probes(3, 2, 8, 500e-9, 650e-9)
        s.step(7)
    np.testing.assert_array_equal(a.field("Ey"), b.field("Ey"))
    for q in range(6):
        np.testing.assert_array_equal(a.face_spectrum(q)[0], b.face_spectrum(q)[0])
    for s in sims:
        s.close()
