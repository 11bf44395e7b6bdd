"""Memory and streams of several contexts: kept blocks are asked back when another context runs out, and tensors of another
torch stream than the context's are read after they are written."""
import numpy as np
import pytest
import torch

from paper_2207_12848_gb300 import Context
from synth import configs
from synth.fields import fibonacci_directions
from synth.mesh import lattice_mesh

pytestmark = pytest.mark.gpu
ROWS = dict(geometry_only=1, schedule="dataflow", lanes_per_task=4)  # one kernel whatever memory is left


def test_another_context_gets_the_kept_blocks(gpu_lib):
    om, w = fibonacci_directions(16, seed=1)
    small, big = lattice_mesh(10), lattice_mesh(64)

    def solve(c, m):
        c.set_mesh(m)
        c.set_directions(om, w)
        c.set_material(np.full((m.n_cells, 1), 0.5), np.ones((m.n_cells, 1)))
        return c.solve(**ROWS)[0]

    with Context(0) as a, Context(0) as b:
        want = solve(b, big)
        solve(b, small)  # b keeps what the large mesh took
        torch.cuda.synchronize()
        torch.cuda.empty_cache()
        held = torch.empty(torch.cuda.mem_get_info(0)[0] - (40 << 20), dtype=torch.uint8, device="cuda")
        try:
            assert np.array_equal(solve(a, big), want)  # about 500 MB
        finally:
            del held
            torch.cuda.empty_cache()
        first = solve(b, small)
        assert np.array_equal(solve(b, big), want) and np.array_equal(solve(b, small), first)


def test_tensors_of_another_stream(gpu_lib):
    p = configs.voronoi_small(3000, n_dir=6, n_groups=2, seed=61)
    ka, em = (torch.from_numpy(v).cuda() for v in (p.kappa_abs, p.emissivity))
    side = torch.cuda.Stream()
    for own in (None, torch.cuda.Stream()):
        with Context(0, own.cuda_stream if own else None) as c:
            c.set_mesh(p.mesh)
            c.set_directions(p.omega, p.weight)
            c.set_material(p.kappa_abs, p.emissivity)
            J, Gamma = c.solve()[:2]
            gk, ge = c.adjoint(dl_dJ=np.ones_like(J))[:2]
            torch.cuda.synchronize()
            with torch.cuda.stream(side):
                for _ in range(3):
                    torch.cuda._sleep(20_000_000)  # about 10 ms
                    k, e = 1.0 * ka, 1.0 * em
                    c.set_material(k, e)
                    del k, e
                    junk = [torch.full_like(ka, 1e6) for _ in range(4)]  # may take the freed tensors' memory
                    out = [torch.full_like(ka, -1.0) for _ in range(4)]
                    torch.cuda._sleep(20_000_000)
                    one = torch.ones_like(ka)
                    c.solve_dev(out[0], out[1])
                    c.adjoint_dev(out[2], out[3], dl_dJ=one)
                    for got, want in zip(out, (J, Gamma, gk, ge)):
                        assert np.array_equal(got.cpu().numpy(), want)
                    del junk
