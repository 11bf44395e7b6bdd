"""The boundary tally under scheme (b), where n.Omega of a chosen vacuum face is all rounding."""
import math

import numpy as np
import pytest

from synth.mesh import FACE_BOUNDARY, Mesh

pytestmark = pytest.mark.gpu

# Omega and n with ((nx ox) + (ny oy)) + (nz oz) > 0 in separately rounded FP64 (the classification: an outflow face), while
# the sum by fused multiply-adds is negative
PAIRS = [([-0.22627306291421131, -0.9703309965542657, 0.08519541141063239], [0.7125299344047463, -0.10524864277676954, 0.6937029737364659]),
         ([0.14095036707748562, 0.7227371838544171, -0.6765973374873039], [-0.3425066420046253, 0.6768167408639206, 0.6516197506744681]),
         ([0.9718938109556724, 0.2352912259104958, -0.007775553716339409], [-0.1745493079755488, 0.7423695418532793, 0.646853926643264]),
         ([0.7191537736360519, -0.27152569035245727, -0.6396027277487546], [-0.35586478292452867, -0.9345312845351839, -0.003396247796832482])]


@pytest.mark.parametrize("inflow", [False, True])
@pytest.mark.parametrize("n", [1, 2, 3, 8])
@pytest.mark.parametrize("pair", range(len(PAIRS)))
def test_share_of_a_grazing_face_escapes(ctx, pair, n, inflow):
    # one cell: faces +-n1 (grazing), +-Omega and +-n3; every chosen face is a vacuum face, so what is not absorbed escapes
    o, n1 = (np.array(v) for v in PAIRS[pair])
    assert (n1[0] * o[0] + n1[1] * o[1]) + n1[2] * o[2] > 0
    n3 = np.cross(o, n1) + 0.5 * o
    n3 /= np.linalg.norm(n3)
    normal = np.array([n1, -n1, o, -o, n3, -n3])
    m = Mesh(volume=np.array([1.0]), face_cells=np.array([[0, -1]] * 6, np.int32), area=np.array([1.0, 1.0, 2.0, 2.0, 1.5, 1.5]),
             normal=normal, flags=np.full(6, FACE_BOUNDARY, np.uint8))
    ctx.set_mesh(m)
    ctx.set_directions(o[None], np.array([4 * math.pi]))
    ctx.set_material(np.array([[0.5]]), np.array([[2.0]]), boundary_inflow=np.linspace(0.5, 1.0, 6)[:, None] if inflow else None)
    J, _, st, _ = ctx.solve(precision=64, transport=n)
    # P = sum of A n.Omega over the outflow faces; the whole outflow P I escapes
    t = (normal[:, 0] * o[0] + normal[:, 1] * o[1]) + normal[:, 2] * o[2]
    P = (m.area * t)[t > 0].sum()
    assert abs(st["escaped"] - 4 * math.pi * P * J[0, 0]) <= 1e-13 * st["escaped"]  # a dozen roundings of 2^-53
    assert abs(st["defect"]) <= 1e-13
