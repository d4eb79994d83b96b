"""The launch that mb_step takes: told whatever selected it, set on any grid
that takes it, the same bits from each; a read answer set again, here or on
another context, is the same launch."""
import numpy as np
import pytest

from parity_util import DT, DX, make_pair, params_kw

pytestmark = pytest.mark.gpu

STATE = ("Ex", "Ey", "Ez", "Hx", "Hy", "Hz", "Px", "Py", "Pz", "Jx", "Jy", "Jz", "N1", "N2", "N3")
TWO, SINGLE, MANY = 0, 1, 2
TILES = [(32, 4), (32, 8), (64, 4), (64, 8)]


@pytest.fixture
def used_memory():
    """Device memory that holds NaNs when it is handed out."""
    from paper_0809_1547_gb300.binding import mb_debug_fill_alloc
    mb_debug_fill_alloc(0xff)
    yield
    mb_debug_fill_alloc(-1)


def _setup(grid, npml, cls=None):
    from paper_0809_1547_gb300 import inputs
    from paper_0809_1547_gb300.binding import MBSimulation, mb_default_params
    eps, gain = inputs.random_small(grid, seed=sum(grid), npml=npml, d_cells=4.0)
    g = MBSimulation(grid, DX, DT, mb_default_params(npml=npml))
    g.set_material(eps, gain, 4e24, 1e13)
    g.set_seed(77)
    # near the end of a row, where its padding begins
    g.set_source((grid[0] - npml - 2, grid[1] // 2, grid[2] // 2), 1, 532e-9, 1.0e-15, 0.4e-15, 1e9)
    for x in (grid[0] - 1, grid[0] // 2, 0):
        g.add_point_probe((x, grid[1] // 2, grid[2] // 2), 9, 480e-9, 700e-9)
    return g


def _snapshot(g):
    out = {f: g.field(f) for f in STATE}
    for w in range(3):
        out[f"psi{w}"] = g.cpml(w)
    for q in range(3):
        out[f"probe{q}"] = g.probe_spectrum(q)[0]
    return out, g.flux(), g.energy()[0]


def _assert_same(ref, got, what):
    for k, v in ref[0].items():
        if v is not None:
            np.testing.assert_array_equal(got[0][k], v, err_msg=f"{what} {k}")
    # FP32 partial sums grouped by the launch's tiles
    np.testing.assert_allclose(got[1], ref[1], rtol=1e-5, atol=1e-5 * np.abs(ref[1]).max(), err_msg=what)
    assert got[2] == pytest.approx(ref[2], rel=1e-13, abs=0), what


# rows padded to a multiple of 16 (the material by tensor copies), to a
# multiple of 4 and rows of 4 k cells (the material by plain loads); fewer
# columns than a tile; ragged rows of tiles
@pytest.mark.parametrize("grid,npml", [((157, 13, 9), 4), ((47, 9, 12), 4), ((95, 9, 7), 2), ((51, 9, 12), 4),
                                       ((20, 5, 3), 1), ((50, 6, 5), 0), ((139, 20, 18), 8)])
def test_single_pass_on_any_rows(grid, npml, used_memory):
    g = _setup(grid, npml)
    g.set_step_launch((TWO, 0, 0, 0))
    g.step(3)
    blob = g.save_state()
    g.step(9)
    ref = _snapshot(g)
    for tile, kz in zip(TILES, (1, 3, 5, 64)):
        g.load_state(blob)
        g.set_step_launch((SINGLE,) + tile + (kz,))
        assert g.step_launch() == (SINGLE,) + tile + (kz,)
        assert g.launch_stats()[0] == 2   # the step and the point probes
        g.step(9)   # odd: ends in the other copy
        _assert_same(ref, _snapshot(g), f"{tile} {kz}")
    g.close()


# padded rows (47, 31, 34, 19 cells), rows of 4 k + 1 cells that are not
@pytest.mark.parametrize("grid,npml", [((47, 41, 17), 4), ((31, 26, 23), 4), ((34, 20, 19), 8), ((19, 24, 28), 3),
                                       ((45, 26, 20), 4), ((33, 12, 20), 0)])
def test_many_steps_on_padded_rows(grid, npml, used_memory):
    g = _setup(grid, npml)
    g.set_step_launch((TWO, 0, 0, 0))
    g.step(2)
    blob = g.save_state()
    g.step(67)
    ref = _snapshot(g)
    g.load_state(blob)
    g.set_step_launch((MANY, 0, 0, 1))
    assert g.step_launch() == (MANY, 0, 0, 1)
    before = g.launch_stats()[1]
    for n in (1, 2, 64):
        g.step(n)
    assert g.launch_stats()[1] == before + 3
    _assert_same(ref, _snapshot(g), "many steps")
    g.close()


@pytest.mark.parametrize("grid,launch", [((139, 20, 18), (SINGLE, 32, 4, 6)), ((51, 20, 18), (MANY, 0, 0, 2))])
def test_energy_after_the_adjoint(grid, launch, used_memory):
    from paper_0809_1547_gb300 import inputs
    eps, gain = inputs.random_small(grid, seed=3, npml=4, d_cells=4.0)
    o, g = make_pair(grid, eps, gain, 4e24, 1e13, 0x3E, params_kw(npml=4))
    o.add_source((9, 9, 9), 2, 532e-9, 1.0e-15, 0.4e-15, 1e9)
    g.set_source((9, 9, 9), 2, 532e-9, 1.0e-15, 0.4e-15, 1e9)
    g.set_step_launch(launch)
    for n in (33, 4):
        g.step(n)
        o.step(n)
        assert g.energy()[0] == pytest.approx(o.energy(), rel=2e-5, abs=0)
    g.adjoint_energy_zface(5, 3)
    o.step(5)
    assert g.step_launch() == launch
    assert g.energy()[0] == pytest.approx(o.energy(), rel=2e-5, abs=0)
    g.close()


# the launches outside the single-pass switch's own rule (n_x % 16 == 0)
@pytest.mark.parametrize("grid,launch", [((24, 22, 20), (MANY, 0, 0, 3)), ((51, 20, 18), (SINGLE, 64, 4, 6)),
                                         ((32, 20, 18), (MANY, 0, 0, 4)), ((32, 20, 18), (SINGLE, 32, 8, 6)),
                                         ((33, 20, 18), (TWO, 32, 8, 32))])
def test_a_read_answer_set_again_is_the_same_launch(grid, launch):
    a, b, c = (_setup(grid, 4) for _ in range(3))
    a.set_step_launch(launch)
    told = a.step_launch()
    assert told[0] == launch[0]
    t = a.single_pass()
    assert t[0] == (1 if launch[0] == SINGLE and grid[0] % 16 == 0 else 0)
    a.set_single_pass(t)
    assert a.step_launch() == told
    b.set_step_launch((TWO, 0, 0, 0))
    b.set_single_pass(t)
    assert b.step_launch()[0] == launch[0]
    c.set_step_launch(a.step_launch())
    assert c.step_launch()[0] == launch[0]
    a.set_single_pass((0, 32, 8, 16))   # off is off
    assert a.step_launch()[0] == TWO
    for s in (a, b, c):
        s.close()


def test_refusals():
    from paper_0809_1547_gb300.binding import MB_ERR_ARG, MBError, MBSimulation, mb_default_params
    s = MBSimulation((33, 8, 8), DX, DT, mb_default_params(npml=2))   # neither padded nor a multiple of 4
    big = MBSimulation((96, 96, 96), DX, DT, mb_default_params(npml=2))
    for g in (s, big):
        g.set_step_launch((TWO, 0, 0, 0))
    for g, bad in ((s, (SINGLE, 32, 4, 4)), (s, (3, 0, 0, 1)), (s, (MANY, 0, 0, 0)), (s, (MANY, 0, 0, 65)),
                   (big, (MANY, 0, 0, 4)), (big, (SINGLE, 32, 16, 4)), (big, (SINGLE, 32, 4, 0))):
        with pytest.raises(MBError) as e:
            g.set_step_launch(bad)
        assert e.value.code == MB_ERR_ARG
        assert g.step_launch()[0] == TWO
    big.set_single_pass((0, 0, 0, -4))   # many steps, read from a small grid: the two passes here
    assert big.step_launch()[0] == TWO
    for q in range(5):
        s.add_point_probe((q, 4, 4), 9, 480e-9, 700e-9)
    with pytest.raises(MBError) as e:
        s.set_step_launch((MANY, 0, 0, 4))
    assert e.value.code == MB_ERR_ARG
    s.step(3)
    for g in (s, big):
        g.close()
