"""A sweep that gave up on a wait leaves nothing behind that a later sweep takes for its own: a solve with another material on
the same context is the answer of a new context."""
import numpy as np
import pytest

from paper_2207_12848_gb300 import Context, SweepError
from synth import configs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind", ["vacuum", "scatter", "periodic"])
@pytest.mark.parametrize("kw", [dict(), dict(op_format="lines"), dict(geometry_only=1), dict(precision=64)])
def test_values_of_a_sweep_that_gave_up(gpu_lib, kw, kind):
    # the dataflow schedule reads a value as soon as its sign is this sweep's; the stalled sweep writes many of them
    p = configs.voronoi_small(4000, periodic_box=kind == "periodic", n_dir=8, seed=41, scatter_albedo=0.5 if kind == "scatter" else 0.0)
    kw = dict(schedule="dataflow", tol_scat=0.0, max_it_scat=2, tol_pbc=0.0, max_it_pbc=2, **kw)
    em = p.emissivity[::-1].copy()

    def load(c, e):
        c.set_mesh(p.mesh)
        c.set_directions(p.omega, p.weight)
        c.set_material(p.kappa_abs, e, kappa_scat=p.kappa_scat)

    with Context(0) as c:
        load(c, em)
        want = c.solve(**kw)[0]
    for before in (0, 1, 2):  # sweeps of the buffer before: both signs
        with Context(0) as c:
            load(c, p.emissivity)
            for _ in range(before):
                c.solve(**kw)
            with pytest.raises(SweepError) as e:
                c.solve(debug_stall=1, spin_budget=20000, **kw)
            assert e.value.status == 4
            c.set_material(p.kappa_abs, em, kappa_scat=p.kappa_scat)
            assert np.array_equal(c.solve(**kw)[0], want)
