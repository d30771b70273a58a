"""Small FP64 grids in one launch (warp-level line solves): one to sixteen chunks per line, chunk
edges, items that end inside a row, one cluster and a whole grid of CTAs, many sources per row,
against the FP64 oracle.  Bound: 1e-12 normwise, as for every FP64 step (test_parity_gpu.py).
"""
import numpy as np
import pytest

import oracle
from paper_2602_05017_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d_max", [1e5, 1e7])
@pytest.mark.parametrize("shape", [(1, 1, 1, 1), (2, 1, 3, 32), (8, 9, 7, 1), (16, 17, 15, 3),
                                   (64, 63, 5, 2), (65, 33, 4, 1), (128, 127, 9, 1),
                                   (3, 128, 120, 2), (7, 5, 128, 31), (40, 41, 39, 5)],
                         ids=lambda s: "x".join(map(str, s)))
def test_small_grid_matches_oracle(shape, d_max):
    from paper_2602_05017_gb300 import binding
    nx, ny, nz, ns = shape
    rng = np.random.default_rng(nx + 3 * ny + 5 * nz)
    w = inputs.random_problem(rng, nx, ny, nz, ns, n_agents=max(1, nx * ny * nz // 2),
                              dirichlet=True, D_range=(1e2, d_max))
    ref = oracle.Problem(**w.oracle_kwargs()).step(w.rho0, 3)
    sim = binding.BioFVM.from_workload(w, precision="fp64")
    assert sim.describe() == "cooperative"
    sim.step(1)
    sim.step(2)
    got = sim.density()
    sim.close()
    assert np.abs(got - ref).max() <= 1e-12 * np.abs(ref).max()
