"""Contexts of several threads: the sweeps by direction of different shared-memory plans side by side."""
import threading

import numpy as np
import pytest
import torch

from paper_2207_12848_gb300 import Context, default_opts
from synth import configs
from synth.fields import fibonacci_directions
from synth.mesh import lattice_mesh

pytestmark = pytest.mark.gpu


def test_two_plans_of_one_kernel_in_two_threads(gpu_lib):
    # the same kernel (1 group, FP32, levels of few slices) with plans of other sizes; every launch has to be accepted
    p, small = configs.voronoi_small(2500, n_dir=6, seed=1), lattice_mesh(4)
    ones = np.ones((small.n_cells, 1))
    probs = [(p.mesh, p.omega, p.weight, p.kappa_abs, p.emissivity), (small, *fibonacci_directions(2, seed=1), ones, ones)]
    errors = []

    def work(mesh, omega, weight, kappa, em):
        try:
            with Context(0, torch.cuda.Stream().cuda_stream) as c:
                c.set_mesh(mesh)
                c.set_directions(omega, weight)
                c.set_material(kappa, em)
                want = c.solve()[0]
                o = default_opts()
                for _ in range(400):
                    J, _, st, _ = c.solve(o)
                    assert st["lanes_used"] == 1 and np.array_equal(J, want)
        except BaseException as e:  # reported by the main thread
            errors.append(e)

    threads = [threading.Thread(target=work, args=q) for q in probs]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
