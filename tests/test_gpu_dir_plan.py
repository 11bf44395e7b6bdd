"""The operator of the sweep by direction: planned once per levelisation, kept per precision and number of groups."""
import numpy as np
import pytest

from synth import configs
from synth.fields import fibonacci_directions
from synth.mesh import Mesh, column_mesh, lattice_mesh

pytestmark = pytest.mark.gpu


def wide_first_level(n_single, n_column):
    """n_single cells that touch nothing, and a column: a narrow mean level, a first level that no ring holds."""
    one, col = lattice_mesh(1), column_mesh(n_column)
    fc = np.tile(one.face_cells, (n_single, 1))
    fc[:, 0] += np.repeat(np.arange(n_single), one.n_faces).astype(np.int32)
    cfc = col.face_cells.copy()
    cfc[cfc >= 0] += n_single
    cat = np.concatenate
    return Mesh(volume=cat([np.tile(one.volume, n_single), col.volume]), face_cells=cat([fc, cfc]),
                area=cat([np.tile(one.area, n_single), col.area]), normal=cat([np.tile(one.normal, (n_single, 1)), col.normal]),
                flags=cat([np.tile(one.flags, n_single), col.flags]))


@pytest.mark.parametrize("precision", [32, 64])
def test_plan_that_does_not_apply_is_made_once(ctx, precision):
    m = wide_first_level(70000, 2000)
    om, w = fibonacci_directions(6, seed=1)
    ctx.set_mesh(m)
    ctx.set_directions(om, w)
    rng = np.random.default_rng(2)
    ctx.set_material(rng.uniform(0.1, 2.0, (m.n_cells, 1)), rng.uniform(0.0, 1.0, (m.n_cells, 1)))
    J, _, first, _ = ctx.solve(precision=precision)
    assert first["lanes_used"] != 1 or first["blocks_per_sm_used"] != 1  # not by direction
    st = [ctx.solve(precision=precision)[2] for _ in range(2)]
    ref = [ctx.solve(precision=precision, schedule="dataflow")[2] for _ in range(2)][1]
    assert st[0]["t_assemble_ms"] == st[1]["t_assemble_ms"] == 0.0
    # what a solve of kept levels launches besides: AUTO's preparation of the source before it looks up its schedule
    assert st[0]["kernel_launches"] == st[1]["kernel_launches"] <= ref["kernel_launches"] + 1
