"""Small-grid launch (many steps per launch, state in shared memory), which
the autotuner picks on small grids: the same bits as the two passes."""
import numpy as np
import pytest

from parity_util import DT, DX

pytestmark = pytest.mark.gpu

STATE = ("Ex", "Ey", "Ez", "Hx", "Hy", "Hz", "Px", "Py", "Pz", "Jx", "Jy", "Jz", "N1", "N2", "N3")


def _pair(grid, npml, dense=False, n_probes=1, faces=0, plane=0, N_a=4e24, src=True):
    """Two contexts of one realization: autotuned, and the default two passes."""
    from paper_0809_1547_gb300 import inputs
    from paper_0809_1547_gb300.binding import MBSimulation, mb_default_params
    eps, gain = inputs.random_small(grid, seed=5, npml=npml, d_cells=4.0)
    if dense:
        eps = eps + np.linspace(0.0, 1.0, eps.size, dtype=np.float32).reshape(eps.shape)
    out = []
    for _ in range(2):
        s = MBSimulation(grid, DX, DT, mb_default_params(npml=npml))
        s.set_material(eps, gain, N_a, 1e13)
        s.set_seed(0x51A11)
        for q in range(n_probes):
            s.add_point_probe((grid[0] // 2, grid[1] // 2, (grid[2] // 2 + q) % grid[2]), 33, 475e-9, 705e-9)
        if faces:
            s.add_face_probes(3, faces, 8, 500e-9, 650e-9)
        if plane:
            s.add_plane_probe(grid[2] // 2, plane, 2, 500e-9, 650e-9)
        if src:
            s.set_source(tuple(v // 3 for v in grid), 1, 532e-9, 1.0e-15, 0.4e-15, 1e9)
        out.append(s)
    out[0].autotune()
    return out


def _same(a, b):
    assert a.n == b.n
    for f in STATE:
        np.testing.assert_array_equal(a.field(f), b.field(f), err_msg=f)
    for w in range(3):
        ca, cb = a.cpml(w), b.cpml(w)
        assert (ca is None) == (cb is None)
        if ca is not None:
            np.testing.assert_array_equal(ca, cb)
    for q in a.probe_nfreq:
        np.testing.assert_array_equal(a.probe_spectrum(q)[0], b.probe_spectrum(q)[0])
    # face energies: FP32 partial sums grouped otherwise
    np.testing.assert_allclose(a.flux(), b.flux(), rtol=1e-5, atol=1e-5 * np.abs(b.flux()).max())


def _launches(s, n):
    before = s.launch_stats()[1]
    s.step(n)
    return s.launch_stats()[1] - before


# boxes of one cell per axis, blocks of one plane, odd edges; more items than
# threads per block; no CPML; CPML slabs meeting in the middle
@pytest.mark.parametrize("grid,npml", [((24, 22, 20), 4), ((33, 41, 17), 4), ((17, 5, 3), 0), ((16, 16, 16), 8),
                                       ((45, 41, 43), 8), ((32, 1, 24), 0), ((7, 90, 31), 3)])
def test_small_grid_equals_two_passes(grid, npml):
    a, b = _pair(grid, npml)
    # a single step (the two passes' launches), an odd count (the state in the
    # other copy), whole launches and a remainder
    _launches(a, 1)
    assert _launches(a, 33) == 1
    assert _launches(a, 100) == 2
    b.step(134)
    _same(a, b)
    assert _launches(a, 64) == 1
    b.step(64)
    _same(a, b)
    for s in (a, b):
        s.close()


def test_small_grid_dense_map_probes_and_read_outs_between():
    a, b = _pair((29, 26, 23), 4, dense=True, n_probes=4, faces=4, plane=3)
    for n in (1, 2, 3, 9, 30):
        a.step(n)
        b.step(n)
        assert a.energy()[0] == pytest.approx(b.energy()[0], rel=1e-13)
    _same(a, b)
    for q in range(6):
        np.testing.assert_allclose(a.face_spectrum(q)[0], b.face_spectrum(q)[0], rtol=1e-12)
    np.testing.assert_array_equal(a.plane_mode_map(0, 1), b.plane_mode_map(0, 1))
    # a state saved from one continues in the other; a step back is a step back
    blob = a.save_state()
    a.step(10)
    b.step(10)
    a.load_state(blob)
    a.step(10)
    _same(a, b)
    # field writes, and more probes than the launch takes (the two passes then)
    for s in (a, b):
        s.set_field("Ez", np.ones(s.shape, np.float32) * (s.field("Ez") != 0))
        s.add_point_probe((3, 3, 3), 33, 475e-9, 705e-9)
        s.step(7)
    _same(a, b)
    for s in (a, b):
        s.close()


def test_small_grid_without_gain_and_adjoint_after():
    a, b = _pair((24, 20, 22), 4, N_a=0.0)
    assert _launches(a, 33) == 1
    b.step(33)
    _same(a, b)
    Ja, ga, _ = a.adjoint_energy_zface(12, 5)
    Jb, gb, _ = b.adjoint_energy_zface(12, 5)
    assert Ja == pytest.approx(Jb, rel=1e-12, abs=0)
    np.testing.assert_array_equal(ga.cpu().numpy(), gb.cpu().numpy())
    assert _launches(a, 15) == 1
    b.step(15)
    _same(a, b)
    for s in (a, b):
        s.close()
