"""FP32 intensities that overflow: infinite and NaN changes do not keep an iteration from stopping."""
import numpy as np
import pytest

from paper_2207_12848_gb300 import Context
from synth import configs
from synth.mesh import concat_meshes

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("graph", [0, 1])
def test_source_iteration_beside_an_overflowing_mesh(ctx, graph):
    # two meshes that share nothing; the sources of the second are above the largest FP32 number
    p, q = (configs.voronoi_small(n, n_dir=6, seed=n, scatter_albedo=0.5) for n in (700, 300))
    kw = dict(precision=32, max_it_scat=200, use_graph=graph)

    def solve(c, mesh, parts):
        c.set_mesh(mesh)
        c.set_directions(p.omega, p.weight)
        c.set_material(*(np.concatenate([getattr(x, k) for x in parts]) for k in ("kappa_abs", "emissivity")),
                       kappa_scat=np.concatenate([x.kappa_scat for x in parts]))
        return c.solve(**kw)

    J, _, st, s = solve(ctx, p.mesh, [p])
    assert s == 0
    q.emissivity = np.where(q.emissivity > 0, 1e300, 0.0)
    J2, _, st2, s2 = solve(ctx, concat_meshes([p.mesh, q.mesh]), [p, q])
    assert s2 == 0 and np.isinf(J2[p.mesh.n_cells:]).any()
    assert np.array_equal(J2[:p.mesh.n_cells], J) and st2["it_scat"] == st["it_scat"]


def test_transposed_iteration_beside_an_overflowing_mesh(ctx):
    # the loss gradient of the second mesh is above the largest FP32 number: its lambda is infinite or NaN
    p, q = (configs.voronoi_small(n, n_dir=6, seed=n, scatter_albedo=0.5) for n in (700, 300))
    rng = np.random.default_rng(5)
    dj = [rng.uniform(0.5, 1.0, x.kappa_abs.shape) for x in (p, q)]
    dj[1][:] = 1e300
    out = []
    for parts, d in (([p], dj[:1]), ([p, q], dj)):
        ctx.set_mesh(concat_meshes([x.mesh for x in parts]))
        ctx.set_directions(p.omega, p.weight)
        ctx.set_material(*(np.concatenate([getattr(x, k) for x in parts]) for k in ("kappa_abs", "emissivity")),
                         kappa_scat=np.concatenate([x.kappa_scat for x in parts]))
        out.append(ctx.adjoint(dl_dJ=np.concatenate(d), precision=32, max_it_scat=5, tol_scat=0.0, allow_not_converged=True))
    n = p.mesh.n_cells
    assert np.array_equal(out[1][1][:n], out[0][1])
    assert not np.isnan(out[1][-1]["res_pbc"])
