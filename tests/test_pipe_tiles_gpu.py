"""The tile of every axis is the one its case is here for, in FP32 and 16-bit storage, against the
FP64 oracle on the same (rounded) field: 24-line tiles on aligned and padded rows, even and odd
substrate counts, and 16-bit fields whose full chunks at a line's ends run unclamped, beside
Dirichlet faces.

Bounds: FP32 normwise 1e-5 (test_parity_gpu.py); 16-bit storage 4 s u + 1e-5 after s steps
(test_storage16_gpu.py).  d_range as in test_pipe_pairs_gpu.py: "varying" has no interior chunks.
"""
import numpy as np
import pytest

import oracle
from paper_2602_05017_gb300 import inputs
from test_storage16_gpu import UNIT_ROUNDOFF, as_f64, rounded

pytestmark = pytest.mark.gpu

N, M = "cw32/m16", "cw24/m48"
CASES = [
    ("fp32", (16, 8, 1000, 2), (N, N, M)), ("fp32", (12, 4, 900, 2), (N, N, M)),
    ("fp32", (20, 8, 760, 6), (N, N, M)), ("fp32", (8, 8, 720, 8), (N, N, M)),
    ("fp32", (4, 900, 5, 1), (N, M, N)), ("fp32", (13, 1000, 3, 2), (N, M, N)),
    ("fp32", (4, 730, 3, 1), (N, "cw32/m48", N)), ("fp32", (9, 8, 1000, 3), (N, N, "cw16/m16")),
    ("bf16", (48, 32, 16, 8), (N, N, N)), ("fp16", (64, 32, 48, 2), (N, N, N)),
    ("fp16", (16, 33, 47, 3), (N, N, N)), ("bf16", (8, 17, 31, 5), (N, N, N)),
    ("fp16", (32, 48, 16, 1), (N, N, N)), ("bf16", (8, 1200, 2, 8), (N, "cw16/m16", N)),
    ("fp16", (8, 4, 1300, 2), (N, N, "cw16/m24")), ("bf16", (8, 4, 912, 7), (N, N, M)),
]


@pytest.mark.parametrize("d_range", [(1e2, 1e5), (1e2, 1e7)], ids=["interior", "varying"])
@pytest.mark.parametrize("prec, shape, tiles", CASES,
                         ids=[f"{p}-{'x'.join(map(str, s))}" for p, s, _ in CASES])
def test_tiles_match_oracle(prec, shape, tiles, d_range):
    from paper_2602_05017_gb300 import binding
    nx, ny, nz, ns = shape
    rng = np.random.default_rng(nx + 31 * ny + 7 * ns)
    w = inputs.random_problem(rng, nx, ny, nz, ns, n_agents=max(1, nx * ny * nz // 20),
                              dirichlet=True, D_range=d_range)
    if prec == "fp32":
        rho, start, bound = w.rho0.astype(np.float32), w.rho0, 1e-5
    else:
        t, start = rounded(w.rho0, prec)
        rho, bound = t.cuda(), 8 * UNIT_ROUNDOFF[prec] + 1e-5
    ref = oracle.Problem(**w.oracle_kwargs()).step(start, 2)
    sim = binding.BioFVM(w.nx, w.ny, w.nz, w.ns, w.dx, w.dt, w.D, w.lam, w.dirichlet_on,
                         w.dirichlet_value, precision=prec)
    assert sim.describe().split()[:3] == [f"{a}=pipe/{t}" for a, t in zip("xyz", tiles)]
    sim.set_sources(w.voxel, w.secretion, w.target, w.uptake, w.weight)
    sim.set_density(rho)
    sim.step(2)
    got = as_f64(sim.density())
    sim.close()
    assert np.abs(got - ref).max() <= bound * np.abs(ref).max()
