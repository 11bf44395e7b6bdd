"""The per-direction sweep (one block per direction, the library's choice on narrow levels) against the sweep
over warp packets on the same context. In FP32 both add a task's entries in the same tree, so every intensity
is equal bit for bit; in FP64 the trees differ from the mesh-row kernel's order by rounding (1e-12)."""
import numpy as np
import pytest

from paper_2207_12848_gb300 import Context
from synth import configs
from synth.fields import fibonacci_directions
from synth.mesh import column_mesh, lattice_mesh, star_mesh

pytestmark = pytest.mark.gpu
LEVEL = 1  # schedule_used of the per-direction sweep: barriers between levels


def load(ctx, p):
    ctx.set_mesh(p.mesh)
    ctx.set_directions(p.omega, p.weight)
    ctx.set_material(p.kappa_abs, p.emissivity, kappa_scat=p.kappa_scat, boundary_inflow=p.boundary_inflow)


def both(ctx, n_dir, equal=True, **kw):
    J, G, st, _ = ctx.solve(**kw)
    I = [ctx.intensity(d) for d in range(n_dir)]
    J0, G0, st0, _ = ctx.solve(schedule="dataflow", **kw)
    I0 = [ctx.intensity(d) for d in range(n_dir)]
    assert st0["schedule_used"] == 2
    for a, b in [(J, J0), (G, G0)] + list(zip(I, I0)):
        if equal:
            assert np.array_equal(a, b)
        else:
            assert np.max(np.abs(a - b)) <= 1e-12 * np.max(np.abs(b))
    return st


@pytest.mark.parametrize("law,transport", [("balance", 0), ("exp", 0), ("balance", 3), ("exp", 1)])
@pytest.mark.parametrize("G", [1, 2, 4])
@pytest.mark.parametrize("kind", ["inflow", "periodic", "scatter"])
def test_equal_to_packets(ctx, kind, G, law, transport):
    p = configs.voronoi_small(3500, periodic_box=kind == "periodic", n_dir=9, n_groups=G, seed=200 + G, n_src=8,
                              scatter_albedo=0.5 if kind == "scatter" else 0.0, bc_inflow=kind == "inflow")
    load(ctx, p)
    st = both(ctx, 9, law=law, transport=transport, tol_scat=0.0, max_it_scat=3, tol_pbc=0.0, max_it_pbc=3)
    assert st["schedule_used"] == LEVEL and st["kernel_used"] == 7


@pytest.mark.parametrize("n", [33, 500, 20000, 90000])
def test_sizes(ctx, n):
    # from levels of a few tasks to levels of several slices (rounds of one to seven worker warps); values leave the ring
    p = configs.voronoi_small(n, periodic_box=n >= 500, n_dir=5, n_groups=4 if n >= 20000 else 1, seed=n, n_src=3)
    load(ctx, p)
    assert both(ctx, 5, tol_pbc=0.0, max_it_pbc=2)["schedule_used"] == LEVEL


def test_more_directions_than_blocks(ctx):
    # blocks take several directions: rings and slots carry over
    p = configs.voronoi_small(700, periodic_box=True, n_dir=300, seed=5)
    load(ctx, p)
    assert both(ctx, 300, tol_pbc=0.0, max_it_pbc=2)["schedule_used"] == LEVEL


@pytest.mark.parametrize("arms", [30, 64, 65])
def test_long_rows(ctx, arms):
    # tasks of more entries than a slice's quads in registers hold; a row of more than 64 sides takes the packets
    m = star_mesh(arms, seed=arms)
    om, w = fibonacci_directions(24, seed=3)
    ctx.set_mesh(m)
    ctx.set_directions(om, w)
    eps = np.zeros((m.n_cells, 1))
    eps[0] = 1.0
    ctx.set_material(np.full((m.n_cells, 1), 2.0), eps, boundary_inflow=np.random.default_rng(1).uniform(0.1, 1.0, (arms, 1)))
    st = both(ctx, 24)
    if arms <= 64:
        assert st["schedule_used"] == LEVEL and st["lanes_used"] == 1
    else:
        assert st["lanes_used"] >= 32  # the packets


def test_lattice_column_and_wide_levels(ctx):
    # exact ties; one cell; one task per level; and levels too wide for one block, which take the packets
    om, w = fibonacci_directions(6, seed=1)
    for m, narrow in ((lattice_mesh(1), True), (column_mesh(2), True), (lattice_mesh(12), True), (column_mesh(300), True), (lattice_mesh(40), False)):
        ctx.set_mesh(m)
        ctx.set_directions(om, w)
        rng = np.random.default_rng(2)
        ctx.set_material(rng.uniform(0.1, 2.0, (m.n_cells, 2)), rng.uniform(0.0, 1.0, (m.n_cells, 2)))
        st = both(ctx, 6)
        assert (st["lanes_used"] == 1) == narrow


def test_material_without_inflow_after_one_with(ctx):
    # the operator stays; its boundary entries then read nothing
    p = configs.voronoi_small(2000, n_dir=6, seed=8, bc_inflow=True)
    load(ctx, p)
    both(ctx, 6)
    ctx.set_material(p.kappa_abs, p.emissivity)
    both(ctx, 6)
    ctx.set_material(np.repeat(p.kappa_abs, 2, 1), np.repeat(p.emissivity, 2, 1))  # other widths rebuild it
    both(ctx, 6)


@pytest.mark.parametrize("G", [1, 2, 4])
@pytest.mark.parametrize("kind", ["inflow", "periodic", "scatter"])
def test_fp64(ctx, kind, G):
    p = configs.voronoi_small(3000, periodic_box=kind == "periodic", n_dir=7, n_groups=G, seed=220 + G, n_src=8,
                              scatter_albedo=0.5 if kind == "scatter" else 0.0, bc_inflow=kind == "inflow")
    load(ctx, p)
    st = both(ctx, 7, equal=False, precision=64, tol_scat=0.0, max_it_scat=3, tol_pbc=0.0, max_it_pbc=3)
    assert st["schedule_used"] == LEVEL


@pytest.mark.parametrize("precision", [32, 64])
@pytest.mark.parametrize("G", [1, 2])
@pytest.mark.parametrize("kind", ["vacuum", "periodic", "scatter"])
def test_transposed(ctx, kind, G, precision):
    p = configs.voronoi_small(3000, periodic_box=kind == "periodic", n_dir=7, n_groups=G, seed=240 + G, n_src=8,
                              scatter_albedo=0.5 if kind == "scatter" else 0.0)
    load(ctx, p)
    rng = np.random.default_rng(4)
    kw = dict(dl_dJ=rng.normal(size=p.kappa_abs.shape), dl_dGamma=rng.normal(size=p.kappa_abs.shape), precision=precision,
              with_kappa_scat=True, allow_not_converged=True, tol_scat=0.0, max_it_scat=3, tol_pbc=0.0, max_it_pbc=3)
    a, b = ctx.adjoint(**kw), ctx.adjoint(schedule="dataflow", **kw)
    assert a[-1]["schedule_used"] == LEVEL and b[-1]["schedule_used"] == 2
    for x, y in zip(a[:3], b[:3]):
        if precision == 32:
            assert np.array_equal(x, y)
        else:
            assert np.max(np.abs(x - y)) <= 1e-12 * np.max(np.abs(y))


def test_two_contexts_side_by_side(ctx):
    p = configs.voronoi_small(2500, periodic_box=True, n_dir=8, seed=12)
    load(ctx, p)
    a = ctx.solve()[0]
    with Context(0) as other:
        load(other, p)
        assert np.array_equal(other.solve()[0], a) and np.array_equal(ctx.solve()[0], a)
