"""The sweep by direction when a wait for its operator copies gives up: status TIMEOUT, and the next solve on the same
context is right. The copies of one stream stop at a round (debug_stall >= 2), so that the wait for it gives up at once; the copies in
flight still land, and every wait stays bounded."""
import numpy as np
import pytest

from paper_2207_12848_gb300 import SweepError
from synth import configs

pytestmark = pytest.mark.gpu


# the first copies (before any round is summed), those of the first turn of the slots, one past it, one far into the
# direction; control words (0) and entries (1); one block per direction, and blocks that take several
@pytest.mark.parametrize("n_dir", [5, 200])
@pytest.mark.parametrize("stream", [0, 1])
@pytest.mark.parametrize("copy", [0, 1, 5, 9, 60])
def test_copy_wait_gives_up(ctx, copy, stream, n_dir):
    p = configs.voronoi_small(2500, n_dir=n_dir, n_groups=2, seed=31, bc_inflow=True)
    ctx.set_mesh(p.mesh)
    ctx.set_directions(p.omega, p.weight)
    ctx.set_material(p.kappa_abs, p.emissivity, boundary_inflow=p.boundary_inflow)
    for precision in (32, 64):
        J, _, st, _ = ctx.solve(precision=precision)
        assert st["lanes_used"] == 1 and st["depth_max"] > 80  # by direction; a round or more per level
        with pytest.raises(SweepError) as e:
            ctx.solve(precision=precision, debug_stall=2 + 2 * copy + stream)
        assert e.value.status == 4
        for _ in range(2):
            J1, _, st, s = ctx.solve(precision=precision)
            assert s == 0 and st["lanes_used"] == 1 and np.array_equal(J, J1)


def test_copy_past_the_last_is_waited_for(ctx):
    p = configs.voronoi_small(600, n_dir=4, n_groups=2, seed=32)
    ctx.set_mesh(p.mesh)
    ctx.set_directions(p.omega, p.weight)
    ctx.set_material(p.kappa_abs, p.emissivity)
    J = ctx.solve()[0]
    assert np.array_equal(ctx.solve(debug_stall=2 + 2 * 100000)[0], J)
