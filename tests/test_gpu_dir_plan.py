"""The operator of the sweep by direction: planned once per levelisation, kept per precision and number of groups."""
import numpy as np
import pytest
import torch

from paper_2207_12848_gb300 import Context
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


def load(ctx, p):
    ctx.set_mesh(p.mesh)
    ctx.set_directions(p.omega, p.weight)
    ctx.set_material(p.kappa_abs, p.emissivity)


def test_calls_of_two_precisions_take_turns(gpu_lib):
    # a solve and an adjoint in FP32 and in FP64 on one context: each finds its operator again, and answers as on a context of its own
    p = configs.voronoi_small(6000, n_dir=12, n_groups=2, seed=51)
    g = np.random.default_rng(3).normal(size=p.kappa_abs.shape)
    want = {}
    for precision in (32, 64):
        with Context(0) as c:
            load(c, p)
            want[precision] = c.solve(precision=precision)[0], c.adjoint(dl_dJ=g, precision=precision)[:2]
    with Context(0) as c:
        load(c, p)
        for turn in range(3):
            for precision in (32, 64):
                J, _, st, _ = c.solve(precision=precision)
                gk, ge, sa = c.adjoint(dl_dJ=g, precision=precision)
                assert st["lanes_used"] == 1 and sa["schedule_used"] == 1
                assert (st["t_assemble_ms"] == 0.0) == (sa["t_assemble_ms"] == 0.0) == (turn > 0)
                assert np.array_equal(J, want[precision][0])
                assert np.array_equal(gk, want[precision][1][0]) and np.array_equal(ge, want[precision][1][1])


def test_more_kinds_than_are_kept(gpu_lib):
    # six kinds (three numbers of groups, two precisions) in turn: the one not asked for for longest makes room
    p = configs.voronoi_small(3000, n_dir=7, n_groups=4, seed=52, periodic_box=True)
    kinds = [(G, precision) for G in (1, 2, 4) for precision in (32, 64)]
    it = dict(tol_pbc=0.0, max_it_pbc=2)

    def solve(c, G, precision):
        c.set_material(p.kappa_abs[:, :G].copy(), p.emissivity[:, :G].copy())
        return c.solve(precision=precision, **it)

    want = {}
    for k in kinds:
        with Context(0) as c:
            load(c, p)
            want[k] = solve(c, *k)[0]
    with Context(0) as c:
        load(c, p)
        for k in kinds + kinds[::-1] + kinds:
            J, _, st, _ = solve(c, *k)
            assert st["lanes_used"] == 1 and np.array_equal(J, want[k])
        c.set_directions(-p.omega, p.weight)  # other levels: none of the kept ones holds any more
        for k in kinds:
            J, _, st, _ = solve(c, *k)
            assert st["t_assemble_ms"] > 0.0 and not np.array_equal(J, want[k])
        c.set_directions(p.omega, p.weight)
        for k in kinds:
            assert np.array_equal(solve(c, *k)[0], want[k])


def test_kept_operators_make_room(gpu_lib):
    # operators of other calls are given up before a call runs out of memory
    p = configs.voronoi_small(60000, n_dir=48, seed=53)
    kw = dict(precision=64, law="exp", schedule="dataflow")  # reads the mesh rows: about 100 MB more
    with Context(0) as c:
        load(c, p)
        want = c.solve(**kw)[0]
    with Context(0) as c:
        load(c, p)
        first = [c.solve(precision=q)[0] for q in (32, 64)]
        torch.cuda.synchronize()
        free = torch.cuda.mem_get_info(0)[0]
        held = torch.empty(free - (8 << 20), dtype=torch.uint8, device="cuda")
        try:
            assert np.array_equal(c.solve(**kw)[0], want)
        finally:
            del held
            torch.cuda.empty_cache()
        for q, J in zip((32, 64), first):
            assert np.array_equal(c.solve(precision=q)[0], J)


@pytest.mark.parametrize("n,kind,n_dir,fwd,tr", [
    (12, "lattice", 6, True, True), (16, "lattice", 6, True, True), (60000, "voronoi", 6, False, True),
    (60000, "voronoi", 40, True, True), (60000, "periodic", 40, True, True), (24, "lattice", 6, False, False),
    (24, "lattice", 200, False, False)])
def test_fp64_four_values(gpu_lib, n, kind, n_dir, fwd, tr):
    # four FP64 values a task leave room for fewer workers from 77 tasks a level on, and the line for them lies lower the
    # fewer directions there are; forward (four groups) and transposed (two), against the mesh-row kernel. Levels of 51, 89,
    # 97 to 100 and 197 tasks
    if kind == "lattice":
        m = lattice_mesh(n)
        om, w = fibonacci_directions(n_dir, seed=1)
        rng = np.random.default_rng(2)
        ka, em = rng.uniform(0.1, 2.0, (m.n_cells, 4)), rng.uniform(0.0, 1.0, (m.n_cells, 4))
    else:
        p = configs.voronoi_small(n, n_dir=n_dir, n_groups=4, seed=54, n_src=8, periodic_box=kind == "periodic")
        m, om, w, ka, em = p.mesh, p.omega, p.weight, p.kappa_abs, p.emissivity
    it = dict(precision=64, tol_pbc=0.0, max_it_pbc=2, tol_scat=0.0, max_it_scat=2)
    with Context(0) as c:
        c.set_mesh(m)
        c.set_directions(om, w)
        c.set_material(ka, em)
        J, _, st, _ = c.solve(**it)
        assert (st["lanes_used"] == 1 and st["blocks_per_sm_used"] == 1) == fwd
        J0 = c.solve(schedule="dataflow", **it)[0]
        assert np.max(np.abs(J - J0)) <= 1e-12 * np.max(J0)
        c.set_material(ka[:, :2].copy(), em[:, :2].copy())
        g = np.random.default_rng(4).normal(size=(m.n_cells, 2))
        a = c.adjoint(dl_dJ=g, allow_not_converged=True, **it)
        b = c.adjoint(dl_dJ=g, allow_not_converged=True, schedule="dataflow", **it)
        assert a[-1]["schedule_used"] == (1 if tr else 2) and b[-1]["schedule_used"] == 2
        for x, y in zip(a[:2], b[:2]):
            assert np.max(np.abs(x - y)) <= 1e-12 * np.max(np.abs(y))


@pytest.mark.parametrize("n_dir,G,by_dir", [(1, 1, False), (16, 1, True), (1, 2, False), (40, 2, True)])
def test_fp64_few_directions(gpu_lib, n_dir, G, by_dir):
    # 348 tasks a level: one block per direction pays where the mesh rows have many directions to sweep
    m = lattice_mesh(32)
    om, w = fibonacci_directions(n_dir, seed=1)
    rng = np.random.default_rng(3)
    with Context(0) as c:
        c.set_mesh(m)
        c.set_directions(om, w)
        c.set_material(rng.uniform(0.1, 2.0, (m.n_cells, G)), rng.uniform(0.0, 1.0, (m.n_cells, G)))
        J, _, st, _ = c.solve(precision=64)
        assert (st["lanes_used"] == 1 and st["blocks_per_sm_used"] == 1) == by_dir
        J0 = c.solve(precision=64, schedule="dataflow")[0]
        assert np.max(np.abs(J - J0)) <= 1e-12 * np.max(J0)


def test_levels_hold_no_more_than_their_arrays(gpu_lib):
    # 64^3 cells, 64 directions: per task the lists, records, classification and levels (44 bytes) and the intensities (4);
    # the levelisation's words (8) stand in the records' memory once these are made
    m = lattice_mesh(64)
    om, w = fibonacci_directions(64, seed=6)
    tasks = m.n_cells * 64
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    with Context(0) as c:
        c.set_mesh(m)
        c.set_directions(om, w)
        c.set_material(np.full((m.n_cells, 1), 0.5), np.ones((m.n_cells, 1)))
        kw = dict(schedule="dataflow", geometry_only=1, lanes_per_task=4)
        before = torch.cuda.mem_get_info(0)[0]
        J = c.solve(**kw)[0]
        for _ in range(6):  # blocks that nothing asked for are given back
            c.solve(**kw)
        used = before - torch.cuda.mem_get_info(0)[0]
        # besides: 32 padding tasks for each possible level in the list (24 bytes each), tables of levels, per-cell arrays
        extra = 32 * m.n_cells * 24 + 3 * 4 * 64 * 65536 + 100 * m.n_cells
        assert used <= 48 * tasks + extra + (16 << 20)
        assert np.array_equal(c.solve(relevel=1, **kw)[0], J)
        assert before - torch.cuda.mem_get_info(0)[0] <= used


def test_merge_counts_as_levelisation(gpu_lib):
    # the task list of all directions, made when a sweep first needs it, is in the levelisation's time
    p = configs.voronoi_small(20000, n_dir=16, seed=55)
    with Context(0) as c:
        load(c, p)
        assert c.solve()[2]["lanes_used"] == 1  # by direction: no such list
        st = c.solve(schedule="dataflow")[2]
        assert 0.0 < st["t_levelise_ms"] < st["t_total_ms"]
        assert c.solve(schedule="dataflow")[2]["t_levelise_ms"] == 0.0
        c.set_material(p.kappa_abs, p.emissivity)
        c.set_directions(p.omega, p.weight)
        c.solve()
        st = c.adjoint(dl_dJ=np.ones((20000, 1)), schedule="dataflow")[2]
        assert st["t_levelise_ms"] > 0.0
