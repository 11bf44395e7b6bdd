"""The periodic iteration's inflow and its relative change, against sums over the faces on the host."""
import numpy as np
import pytest

from paper_2207_12848_gb300 import Context
from synth import configs

pytestmark = pytest.mark.gpu


def _inflow(p, I):
    """j[c][g] = sum over directions and periodic inflow sides of w A |n.Omega| I_partner; I is [D][N][G]"""
    m = p.mesh
    f = np.nonzero(m.flags & 2)[0]
    j = np.zeros(I.shape[1:])
    c = np.asarray(m.face_cells).reshape(-1, 2)[f]
    for d in range(p.n_dir):
        n, o = m.normal[f], p.omega[d]
        t = (n[:, 0] * o[0] + n[:, 1] * o[1]) + n[:, 2] * o[2]  # the classification's expression and order
        w = (p.weight[d] * m.area[f] * np.abs(t))[:, None]
        for inflow, here, there in ((t < 0, c[:, 0], c[:, 1]), (t > 0, c[:, 1], c[:, 0])):
            np.add.at(j, here[inflow], (w * I[d][there])[inflow])
    return j


# direction counts below, at and above a warp and a block of 128; groups with and without a vector load; 200 cells hold
# less than 2049 periodic cells (one reducing block), 14000 hold more (a cluster)
@pytest.mark.parametrize("n_cells,n_dir,groups,precision", [
    (200, 1, 1, 32), (200, 31, 2, 32), (200, 33, 3, 64), (200, 129, 4, 32), (150, 12, 8, 32), (150, 12, 2, 64),
    (150, 12, 4, 64), (14000, 3, 1, 32)])
def test_inflow_and_change(n_cells, n_dir, groups, precision):
    p = configs.voronoi_small(n_cells, periodic_box=True, n_dir=n_dir, n_groups=groups, seed=n_dir + groups)
    j = []
    for it in (1, 2):
        with Context(0) as c:
            c.set_mesh(p.mesh)
            c.set_directions(p.omega, p.weight)
            c.set_material(p.kappa_abs, p.emissivity)
            st = c.solve(precision=precision, max_it_pbc=it, allow_not_converged=True)[2]
            j.append(_inflow(p, np.stack([c.intensity(d) for d in range(n_dir)])))
    assert st["it_pbc"] == 2
    s = j[0] + j[1]
    e = np.where(s > 0, np.abs(j[1] - j[0]) / np.where(s > 0, s, 1.0), 0.0)
    # both sides sum at most 64 sides of n_dir directions in FP64: each j is good to that many half units of 2^-52, E
    # (a quotient of at most 1) to as many whole ones
    tol = (64 * n_dir + 8) * 2.0 ** -52
    assert abs(st["res_pbc"] - e.max()) <= tol
    assert abs(st["res_pbc_mean"] - e.mean()) <= tol
