"""Sources of small FP64 grids in one launch: none, few and many entries in an item of lines, items
that share a row (more substrates than an item has lines), agents in every voxel and in a clump,
several of them in one voxel, with and without Dirichlet faces, against the FP64 oracle.  Bound:
1e-12 normwise, as for every FP64 step (test_parity_gpu.py).
"""
import numpy as np
import pytest

import oracle
from paper_2602_05017_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dirichlet", [False, True])
@pytest.mark.parametrize("where", ["everywhere", "clump", "few"])
@pytest.mark.parametrize("shape", [(50, 20, 9, 1), (50, 11, 7, 4), (33, 10, 9, 5), (12, 12, 12, 1),
                                   (100, 9, 30, 3), (9, 40, 30, 31), (128, 60, 9, 2)],
                         ids=lambda s: "x".join(map(str, s)))
def test_sources_match_oracle(shape, where, dirichlet):
    from paper_2602_05017_gb300 import binding
    nx, ny, nz, ns = shape
    rng = np.random.default_rng(nx + 3 * ny + 5 * nz)
    nvox = nx * ny * nz
    w = inputs.random_problem(rng, nx, ny, nz, ns, n_agents=1, dirichlet=dirichlet)
    if where == "everywhere":
        voxel = np.concatenate([np.arange(nvox), rng.integers(0, nvox, nvox // 3)])
    elif where == "clump":  # consecutive voxels: five to the row's length in one row
        voxel = np.arange(nvox // 2, nvox // 2 + nx + 5) % nvox
    else:
        voxel = rng.integers(0, nvox, max(1, nvox // 400))
    w.voxel, w.weight = rng.permutation(voxel).astype(np.int64), None
    w.secretion, w.uptake = (rng.uniform(0.0, 5.0, (len(voxel), ns)) for _ in range(2))
    w.secretion[rng.random(w.secretion.shape) < 0.2] = 0.0
    w.target = rng.uniform(0.0, 38.0, (len(voxel), ns))
    ref = oracle.Problem(**w.oracle_kwargs()).step(w.rho0, 3)
    sim = binding.BioFVM.from_workload(w, precision="fp64")
    assert sim.describe() == "cooperative"
    sim.step(3)
    got = sim.density()
    sim.close()
    assert np.abs(got - ref).max() <= 1e-12 * np.abs(ref).max()
