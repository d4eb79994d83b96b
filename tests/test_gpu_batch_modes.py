"""The persistent launch of a batch follows its members' current copy of the
state: after the members' own launches on concurrent streams, which may end
in the second copy, and after an adjoint call on a member, which moves the
state back to the first."""
import numpy as np
import pytest

from parity_util import DT, DX

pytestmark = pytest.mark.gpu

STATE = ("Ex", "Ey", "Ez", "Hx", "Hy", "Hz", "Px", "Jy", "N1", "N2", "N3")
GRIDS = [(48, 21, 19), (51, 19, 23), (33, 27, 20)]   # (sizes no other test uses: tuned here)


def _batch(tuned):
    from paper_0809_1547_gb300 import inputs
    from paper_0809_1547_gb300.binding import MBBatch, mb_default_params
    b = MBBatch(GRIDS, DX, DT, mb_default_params(npml=4))
    for q, grid in enumerate(GRIDS):
        eps, gain = inputs.random_small(grid, seed=q, npml=4, d_cells=4.0)
        b.set_instance(q, eps, gain, 4e24, 1e13, 40 + q)
        b.instances[q].set_source((9, 9, 9), 2, 532e-9, 1.0e-15, 0.4e-15, 1e9)
        if tuned:   # the launches many steps long or in a single pass, where faster
            b.instances[q].autotune()
    if tuned:
        b.instances[0].set_single_pass((1, 32, 4, 8))
    return b


def test_mode_switches_between_odd_step_counts():
    from paper_0809_1547_gb300.binding import MB_BATCH_CONCURRENT, MB_BATCH_PERSISTENT
    a, r = _batch(True), _batch(False)
    r.step(33 + 8 + 1 + 5)
    for mode, n in ((MB_BATCH_CONCURRENT, 33), (MB_BATCH_PERSISTENT, 8), (MB_BATCH_CONCURRENT, 1),
                    (MB_BATCH_PERSISTENT, 5)):
        a.set_mode(mode)
        a.step(n)
    for q in range(len(GRIDS)):
        for f in STATE:
            np.testing.assert_array_equal(a.instances[q].field(f), r.instances[q].field(f), err_msg=f"{q} {f}")
    for b in (a, r):
        b.close()


def test_adjoint_on_a_member_between_calls():
    from paper_0809_1547_gb300.binding import MB_BATCH_CONCURRENT, MB_BATCH_PERSISTENT
    a, r = _batch(True), _batch(False)
    a.set_mode(MB_BATCH_CONCURRENT)
    a.step(33)
    a.set_mode(MB_BATCH_PERSISTENT)
    a.step(2)
    blobs = [s.save_state() for s in a.instances]
    for s, blob in zip(a.instances, blobs):
        s.adjoint_energy_zface(6, 4)
        s.load_state(blob)   # back in step with the batch
    a.step(4)
    r.step(39)
    for q in range(len(GRIDS)):
        for f in STATE:
            np.testing.assert_array_equal(a.instances[q].field(f), r.instances[q].field(f), err_msg=f"{q} {f}")
    for b in (a, r):
        b.close()


@pytest.mark.parametrize("grids", [[(24, 23, 21), (28, 25, 24)], [(48, 40, 44), (51, 47, 40), (40, 44, 36)]])
def test_autotuned_small_members(grids):
    """The trials of a batch of small grids (many steps a launch or two passes,
    all members running) leave the states, and what they pick steps the same."""
    from paper_0809_1547_gb300 import inputs
    from paper_0809_1547_gb300.binding import MB_BATCH_CONCURRENT, MBBatch, mb_default_params
    out = []
    for tuned in (True, False):
        b = MBBatch(grids, DX, DT, mb_default_params(npml=4))
        for q, grid in enumerate(grids):
            eps, gain = inputs.random_small(grid, seed=q, npml=4, d_cells=4.0)
            b.set_instance(q, eps, gain, 4e24, 1e13, 40 + q)
            b.instances[q].set_source((9, 9, 9), 2, 532e-9, 1.0e-15, 0.4e-15, 1e9)
            b.instances[q].add_point_probe((9, 9, 10), 9, 480e-9, 700e-9)
        b.step(5)
        if tuned:
            b.autotune()
            b.set_mode(MB_BATCH_CONCURRENT)
        for n in (1, 3, 64, 33):
            b.step(n)
        b.synchronize()
        out.append(b)
    a, r = out
    for q in range(len(grids)):
        assert a.instances[q].n == r.instances[q].n == 106
        for f in STATE:
            np.testing.assert_array_equal(a.instances[q].field(f), r.instances[q].field(f), err_msg=f"{q} {f}")
        np.testing.assert_array_equal(a.instances[q].probe_spectrum(0)[0], r.instances[q].probe_spectrum(0)[0])
    for b in out:
        b.close()
