"""Launch shapes tuned on padded rows are not handed to a context of the same
grid whose rows are not padded (no memory was left for it), nor the other way."""
import pytest

from parity_util import DT, DX

pytestmark = pytest.mark.gpu


def _sim(grid, padded):
    from paper_0809_1547_gb300.binding import MBSimulation, mb_debug_fail_alloc, mb_default_params
    mb_debug_fail_alloc(-1 if padded else 0)
    try:
        return MBSimulation(grid, DX, DT, mb_default_params(npml=2))
    finally:
        mb_debug_fail_alloc(-1)


# (sizes no other test tunes)
@pytest.mark.parametrize("grid,first", [((131, 75, 45), True), ((131, 77, 46), False)])
def test_shapes_kept_apart(grid, first):
    a = _sim(grid, first)
    before = a.tuning(), a.step_launch()
    assert before[1][0] == 0   # untuned: two passes
    a.autotune()
    b, c = _sim(grid, not first), _sim(grid, first)
    assert (a.device_bytes() > b.device_bytes()) or not first
    assert (b.tuning(), b.step_launch()) == before          # the other rows: untuned
    assert (c.tuning(), c.step_launch()) == (a.tuning(), a.step_launch())
    if not first:
        a, b = b, a
    a.set_step_launch((1, 32, 4, 8))        # padded
    with pytest.raises(Exception):
        b.set_step_launch((1, 32, 4, 8))    # not
    for s in (a, b, c):
        s.step(3)
        s.close()
