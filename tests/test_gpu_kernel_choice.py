"""Which kernel sweeps what, by what only that kernel reports (by direction: one lane and one block per SM; packets: 32 lanes per
packet of a warp step), and the forms that no other test pins to their kernel."""
import numpy as np
import pytest

import oracle
from synth import configs
from synth.fields import fibonacci_directions
from synth.mesh import lattice_mesh, star_mesh

pytestmark = pytest.mark.gpu
PACKED = 7
FP32_TOL = 1e-5


def load(ctx, p):
    ctx.set_mesh(p.mesh)
    ctx.set_directions(p.omega, p.weight)
    ctx.set_material(p.kappa_abs, p.emissivity, kappa_scat=p.kappa_scat, boundary_inflow=p.boundary_inflow)


def by_direction(st):
    return st["lanes_used"] == 1 and st["blocks_per_sm_used"] == 1


def fp32_err(x, ref):
    m = ref >= 1e-30 * ref.max()
    return float(np.max(np.abs(x[m] - ref[m]) / ref[m]))


def run_oracle(p, **kw):
    return oracle.solve(p.mesh, p.omega, p.weight, p.kappa_abs, p.emissivity, kappa_scat=p.kappa_scat,
                        bc_inflow=p.boundary_inflow, threads=8, **kw)


def close64(ctx, n_dir, **kw):
    """FP64 by direction against the mesh-row kernel: every intensity within 1e-12 of the largest."""
    J, _, st, _ = ctx.solve(precision=64, **kw)
    I = [ctx.intensity(d) for d in range(n_dir)]
    J0, _, st0, _ = ctx.solve(precision=64, schedule="dataflow", **kw)
    assert by_direction(st) and not by_direction(st0)
    for a, b in [(J, J0)] + list(zip(I, [ctx.intensity(d) for d in range(n_dir)])):
        assert np.max(np.abs(a - b)) <= 1e-12 * np.max(np.abs(b))


@pytest.mark.parametrize("n,n_dir,G,kw", [
    (33, 5, 1, {}), (500, 5, 1, {}), (20000, 5, 4, {}), (90000, 5, 4, {}), (700, 300, 1, {}), (3500, 9, 2, {}),
    (3500, 9, 1, dict(law="exp")), (3500, 9, 4, dict(transport=3)), (3000, 7, 1, dict(precision=64)),
    (3000, 7, 2, dict(precision=64)), (3000, 7, 4, dict(precision=64))])
def test_auto_sweeps_by_direction(ctx, n, n_dir, G, kw):
    p = configs.voronoi_small(n, n_dir=n_dir, n_groups=G, seed=n, n_src=3)
    load(ctx, p)
    assert by_direction(ctx.solve(**kw)[2])
    assert not by_direction(ctx.solve(schedule="level", **kw)[2])


@pytest.mark.parametrize("G,n_dir,by_dir", [(4, 2, False), (4, 16, True), (2, 2, True)])
def test_four_groups_few_directions(ctx, G, n_dir, by_dir):
    # 197 tasks a level; FP32 intensities are the packets' bit for bit on either side of the line
    m = lattice_mesh(24)
    om, w = fibonacci_directions(n_dir, seed=1)
    rng = np.random.default_rng(3)
    ctx.set_mesh(m)
    ctx.set_directions(om, w)
    ctx.set_material(rng.uniform(0.1, 2.0, (m.n_cells, G)), rng.uniform(0.0, 1.0, (m.n_cells, G)))
    J, _, st, _ = ctx.solve()
    assert by_direction(st) == by_dir
    assert np.array_equal(J, ctx.solve(schedule="dataflow", packets_per_step=2)[0])


@pytest.mark.parametrize("kind", ["vacuum", "periodic", "inflow"])
@pytest.mark.parametrize("n", [1, 3])
@pytest.mark.parametrize("G", [1, 2, 4])
def test_fp64_direction_conserving(ctx, G, n, kind):
    # n = 1 has wide levels: 158 tasks at 3000 cells, more than four values take by direction; 66 at 800
    p = configs.voronoi_small(800 if G == 4 and n == 1 else 3000, periodic_box=kind == "periodic", n_dir=7, n_groups=G,
                              seed=230 + G, n_src=8, bc_inflow=kind == "inflow")
    load(ctx, p)
    close64(ctx, 7, transport=n, tol_pbc=0.0, max_it_pbc=3)


@pytest.mark.parametrize("G", [1, 2, 4])
@pytest.mark.parametrize("arms", [20, 31, 36, 64])
def test_fp64_long_tasks(ctx, arms, G):
    # a hub of about arms / 2 entries: 15 and fewer in registers, the others from shared memory
    m = star_mesh(arms, seed=arms)
    om, w = fibonacci_directions(24, seed=3)
    ctx.set_mesh(m)
    ctx.set_directions(om, w)
    eps = np.zeros((m.n_cells, G))
    eps[0] = 1.0
    ctx.set_material(np.full((m.n_cells, G), 2.0), eps, boundary_inflow=np.random.default_rng(1).uniform(0.1, 1.0, (arms, G)))
    close64(ctx, 24)


@pytest.mark.parametrize("use_graph", [1, 0])
@pytest.mark.parametrize("schedule", ["dataflow", "level"])
def test_packets_scattering_iteration(ctx, schedule, use_graph):
    p = configs.voronoi_small(4000, n_dir=12, n_groups=2, seed=77, scatter_albedo=0.5, n_src=8)
    load(ctx, p)
    J, _, st, _ = ctx.solve(precision=32, schedule=schedule, tol_scat=0.0, max_it_scat=6, use_graph=use_graph)
    assert st["kernel_used"] == PACKED and st["lanes_used"] >= 32 and st["it_scat"] == 6
    assert fp32_err(J, run_oracle(p, tol_scat=0.0, max_it_scat=6)["J"]) <= FP32_TOL


def test_packets_on_a_2p18_box(ctx):
    # the packed kernel on the benchmark's periodic box at 2^18 cells, 128 directions: J and Gamma after three periodic
    # iterations against the oracle, in the launch forms the autotuner chooses from
    p = configs.periodic(n_cells=1 << 18)
    load(ctx, p)
    it = dict(tol_pbc=0.0, max_it_pbc=3)
    r = run_oracle(p, **it)
    first = None
    for kw in (dict(schedule="dataflow", packets_per_step=2), dict(schedule="dataflow", packets_per_step=2, blocks_per_sm=3),
               dict(schedule="dataflow", packets_per_step=1), dict(schedule="level", packets_per_step=2)):
        J, Gm, st, _ = ctx.solve(precision=32, **kw, **it)
        assert st["kernel_used"] == PACKED and st["lanes_used"] == 32 * kw["packets_per_step"]
        assert fp32_err(J, r["J"]) <= FP32_TOL and fp32_err(Gm, r["Gamma"]) <= FP32_TOL
        first = J if first is None else first
        assert np.array_equal(J, first)  # every form adds a task's entries in one order
    J, _, st, s = ctx.solve(precision=32, schedule="dataflow", tol_pbc=1e-6, max_it_pbc=200)
    assert s == 0 and abs(st["defect"]) <= 1e-6
