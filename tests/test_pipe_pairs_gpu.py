"""The pipelined FP32 sweep's column pairs: chunk edges, pair classes of every kind of substrate
count, pairs across rows, both tile widths and the longer chunks of long lines, against the FP64
oracle.

FP32 bound: normwise 1e-5, as for every FP32 step (test_parity_gpu.py).  D_range reaches
r = D dt / dx^2 = 250, where the coefficients are nowhere at their interior values, and 0.0025,
where they are from position 1 on.
"""
import numpy as np
import pytest

import oracle
from paper_2602_05017_gb300 import inputs

pytestmark = pytest.mark.gpu

SHAPES = [
    (16, 15, 17, 1), (32, 31, 33, 1), (33, 47, 49, 4),      # around one, two and three chunks
    (64, 48, 80, 2), (48, 65, 64, 8), (40, 30, 50, 6),      # even counts, compiled and general
    (20, 21, 40, 5), (12, 40, 17, 9), (4, 33, 20, 32),      # odd counts, one row per tile
    (11, 4, 37, 1), (7, 8, 70, 3),                          # z tiles whose pairs cross rows
    (700, 3, 8, 4), (8, 704, 2, 1), (4, 2, 1300, 1),        # chunks of 24, 16-line tiles
    (4, 730, 3, 1), (12, 4, 900, 2), (9, 8, 1000, 3),       # chunks of 48, 24 and 16 lines
]


@pytest.mark.parametrize("d_range", [(1e2, 1e5), (1e2, 1e7)], ids=["interior", "varying"])
@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: "x".join(map(str, s)))
def test_pairs_match_oracle(shape, d_range):
    from paper_2602_05017_gb300 import binding
    nx, ny, nz, ns = shape
    rng = np.random.default_rng(nx + 31 * ny + 7 * ns)
    w = inputs.random_problem(rng, nx, ny, nz, ns, n_agents=max(1, nx * ny * nz // 20),
                              dirichlet=True, D_range=d_range)
    ref = oracle.Problem(**w.oracle_kwargs()).step(w.rho0, 2)
    sim = binding.BioFVM.from_workload(w, precision="fp32")
    sim.step(2)
    got = sim.density().astype(np.float64)
    sim.close()
    assert np.abs(got - ref).max() <= 1e-5 * np.abs(ref).max()
