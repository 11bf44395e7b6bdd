"""Calls that run out of device memory: status OOM, and a context that answers the next call as a new one would (no
buffer of the failed call is left half allocated or is given up twice)."""
import numpy as np
import pytest
import torch

from paper_2207_12848_gb300 import Context, SweepError
from synth.fields import fibonacci_directions
from synth.mesh import lattice_mesh

pytestmark = pytest.mark.gpu
MB = 1 << 20
OOM = 5
# one kernel whatever memory is left (the assembled operators need room, and their sums another order)
ROWS = dict(geometry_only=1, schedule="dataflow", lanes_per_task=4)


class Leave:
    """Device memory taken so that `mb` MiB stay free."""

    def __init__(self, mb):
        torch.cuda.synchronize()
        torch.cuda.empty_cache()
        free = torch.cuda.mem_get_info(0)[0]
        if free < 4 * mb * MB:
            pytest.skip("the device is nearly full")
        self.held = torch.empty(free - mb * MB, dtype=torch.uint8, device="cuda")

    def __enter__(self):
        return self

    def __exit__(self, *a):
        del self.held
        torch.cuda.empty_cache()


def material(n, seed):
    rng = np.random.default_rng(seed)
    return rng.uniform(0.1, 2.0, (n, 1)), rng.uniform(0.0, 1.0, (n, 1))


def answer(c, m, om, w, **kw):
    c.set_mesh(m)
    c.set_directions(om, w)
    c.set_material(*material(m.n_cells, 1))
    return c.solve(**ROWS, **kw)[0]


@pytest.mark.parametrize("mb", [20, 45, 70, 110, 160])
def test_mesh_that_does_not_fit(gpu_lib, mb):
    # 2^18 cells take about 190 MB; what is left stops the call at another of its buffers each time
    om, w = fibonacci_directions(6, seed=1)
    small, big = lattice_mesh(14), lattice_mesh(64)
    with Context(0) as c:
        want = answer(c, small, om, w)
    with Context(0) as c:
        answer(c, small, om, w)
        with Leave(mb):
            for _ in range(2):
                with pytest.raises(SweepError) as e:
                    c.set_mesh(big)
                assert e.value.status == OOM
            for _ in range(2):
                assert np.array_equal(answer(c, small, om, w), want)
        c.set_mesh(big)
        assert np.array_equal(answer(c, small, om, w), want)


@pytest.mark.parametrize("kw", [{}, dict(transport=2)])
@pytest.mark.parametrize("mb", [50, 150, 450, 600])
def test_levels_that_do_not_fit(gpu_lib, mb, kw):
    # 32^3 cells, 512 directions: about 0.5 GB of levels; asked for twice, both calls have to refuse
    om, w = fibonacci_directions(512, seed=2)
    m = lattice_mesh(32)
    with Context(0) as c:
        want = answer(c, m, om, w, **kw)
    with Context(0) as c:
        c.set_mesh(m)
        c.set_directions(om, w)
        c.set_material(*material(m.n_cells, 1))
        with Leave(mb):
            for _ in range(2):
                with pytest.raises(SweepError) as e:
                    c.solve(**ROWS, **kw)
                assert e.value.status == OOM
        assert np.array_equal(c.solve(**ROWS, **kw)[0], want)
