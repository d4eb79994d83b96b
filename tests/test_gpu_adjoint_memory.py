"""The adjoint's device memory is the call's own: taken for it, given back
before it returns, and refused without a change of the state."""
import numpy as np
import pytest

from parity_util import DT, DX

pytestmark = pytest.mark.gpu


def _sim():
    from paper_0809_1547_gb300 import inputs
    from paper_0809_1547_gb300.binding import MBSimulation, mb_default_params
    grid = (64, 60, 56)   # 200 stored steps: 1.6 GB
    eps, gain = inputs.random_small(grid, seed=2, npml=4, d_cells=5.0)
    s = MBSimulation(grid, DX, DT, mb_default_params(npml=4))
    s.set_material(eps, gain, 4e24, 1e13)
    s.set_seed(4)
    s.set_source((32, 30, 28), 0, 560e-9, 1.0e-15, 0.4e-15, 5e13)
    s.step(20)
    return s


def test_memory_given_back():
    import torch
    s = _sim()
    s.adjoint_energy_zface(4, 2)   # graphs, kernels and the gradient's own block
    torch.cuda.synchronize()
    held, free = s.device_bytes(), torch.cuda.mem_get_info()[0]
    g = s.adjoint_energy_zface(200, 200)[1]
    del g
    torch.cuda.synchronize()
    assert s.device_bytes() == held
    # 2 MB granules of the driver's own bookkeeping, no more
    assert free - torch.cuda.mem_get_info()[0] <= 8 << 20
    s.close()


def test_out_of_memory_leaves_the_state():
    from paper_0809_1547_gb300.binding import MB_ERR_OOM, MBError, mb_debug_fail_alloc
    s = _sim()
    n, before = s.n, s.save_state()
    mb_debug_fail_alloc(0)
    try:
        with pytest.raises(MBError) as e:
            s.adjoint_energy_zface(12, 5)
    finally:
        mb_debug_fail_alloc(-1)
    assert e.value.code == MB_ERR_OOM
    assert s.n == n
    np.testing.assert_array_equal(np.frombuffer(s.save_state(), np.uint8), np.frombuffer(before, np.uint8))
    s.adjoint_energy_zface(12, 5)
    s.close()
