"""Device memory kept by a context between calls: results do not depend on what a block held before, and it is given back."""
import numpy as np
import pytest
import torch

from paper_2207_12848_gb300 import Context
from synth import configs

pytestmark = pytest.mark.gpu


def _load(ctx, p):
    ctx.set_mesh(p.mesh)
    ctx.set_directions(p.omega, p.weight)
    ctx.set_material(p.kappa_abs, p.emissivity, kappa_scat=p.kappa_scat, boundary_inflow=p.boundary_inflow)


@pytest.mark.parametrize("precision", [32, 64])
def test_reused_blocks(precision):
    # sizes up and down, so that blocks are reused by requests of their own size, a little smaller, and not at all
    probs = [configs.voronoi_small(n, n_dir=6, n_groups=g, seed=n, periodic_box=per, scatter_albedo=a)
             for n, g, per, a in ((600, 2, True, 0.0), (520, 2, False, 0.4), (600, 1, True, 0.0), (3000, 2, False, 0.0))]
    rng = np.random.default_rng(3)
    want = []
    for p in probs:
        with Context(0) as c:
            _load(c, p)
            J, Gam, _, _ = c.solve(precision=precision)
            g = None if p.mesh.periodic else rng.normal(size=J.shape)
            want.append((J, Gam, g, None if g is None else c.adjoint(dl_dJ=g, precision=precision)[:2]))
    with Context(0) as c:
        for k in [0, 1, 0, 2, 1, 3, 1, 0, 3]:
            _load(c, probs[k])
            J, Gam, _, _ = c.solve(precision=precision)
            np.testing.assert_array_equal(J, want[k][0])
            np.testing.assert_array_equal(Gam, want[k][1])
            if want[k][2] is not None:
                for a, b in zip(c.adjoint(dl_dJ=want[k][2], precision=precision)[:2], want[k][3]):
                    np.testing.assert_array_equal(a, b)


def test_memory_is_given_back():
    p = configs.voronoi_small(3000, n_dir=6, seed=1)
    with Context(0) as c:  # what the first context of a process leaves behind (module, events) is not the pool's
        _load(c, p)
        c.solve()
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info(0)[0]
    big = configs.voronoi_small(20000, n_dir=24, n_groups=4, seed=2)
    with Context(0) as c:
        _load(c, big)
        c.solve()
        held = torch.cuda.mem_get_info(0)[0]
        _load(c, p)
        for _ in range(6):  # nothing asks for the large blocks any more
            c.set_material(p.kappa_abs, p.emissivity)
            c.solve()
        assert torch.cuda.mem_get_info(0)[0] > held
    # a slack of 64 MiB for what else uses the GPU's memory through the driver
    assert torch.cuda.mem_get_info(0)[0] >= before - (64 << 20)
