"""The tallies' integer widening of FP32 intensities and their factored sums, against the intensities read
back one direction at a time (converted by the conversion instruction)."""
import math

import numpy as np
import pytest

from synth import configs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("scale", [1.0, 1e-37, 1e-41, 1e-44, 1e30])
@pytest.mark.parametrize("n_dir", [1, 7, 8, 17])
def test_mean_intensity_is_the_sum_of_the_intensities(ctx, scale, n_dir):
    # normal, denormal and zero values (cells upwind of the sources), direction counts around the unrolling of eight
    p = configs.voronoi_small(900, n_dir=n_dir, n_groups=2, seed=n_dir, n_src=2)
    ctx.set_mesh(p.mesh)
    ctx.set_directions(p.omega, p.weight)
    ctx.set_material(p.kappa_abs, p.emissivity * scale)
    J, Gm, st, _ = ctx.solve(precision=32)
    I = np.stack([ctx.intensity(d) for d in range(n_dir)])
    if scale <= 1e-41:
        assert np.any((I > 0) & (I < 1.1754944e-38))
    assert np.any(I == 0)
    ref = (p.weight[:, None, None] * I).sum(0) / (4 * math.pi)
    # n_dir sums and one quotient, each half a unit in the last place (2^-53)
    assert np.all(np.abs(J - ref) <= (n_dir + 3) * 2.0 ** -52 * ref)
    ref = p.kappa_abs * p.mesh.volume[:, None] * 4 * math.pi * J
    assert np.all(np.abs(Gm - ref) <= 2.0 ** -50 * ref)
