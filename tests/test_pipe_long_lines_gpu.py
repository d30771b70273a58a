"""Pipelined sweeps of long lines at odd substrate counts, whose coefficients are staged per
substrate ("split"), against the FP64 oracle on the same (rounded) field.

Bounds: FP32 normwise 1e-5 (test_parity_gpu.py); 16-bit storage 4 s u + 1e-5 after s steps
(test_storage16_gpu.py).
"""
import numpy as np
import pytest

import oracle
from paper_2602_05017_gb300 import inputs
from test_storage16_gpu import UNIT_ROUNDOFF, as_f64, rounded

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec, shape, axis, tile", [
    ("fp32", (1072, 4, 4, 5), 0, "cw16/m24/split"), ("fp32", (284, 4, 5, 31), 0, "cw32/m24/split"),
    ("fp32", (4, 1256, 3, 3), 1, "cw16/m24/split"), ("fp32", (4, 3, 1408, 3), 2, "cw16/m24/split"),
    ("fp16", (1256, 8, 4, 7), 0, "cw16/m24/split"), ("bf16", (8, 1000, 4, 9), 1, "cw16/m24/split"),
    ("fp16", (8, 4, 448, 25), 2, "cw32/m24/split"), ("bf16", (448, 4, 4, 25), 0, "cw32/m24/split"),
], ids=lambda v: "x".join(map(str, v)) if isinstance(v, tuple) else None)
@pytest.mark.parametrize("d_range", [(1e2, 1e5), (1e2, 1e7)], ids=["interior", "varying"])
def test_split_coefficients_match_oracle(prec, shape, axis, tile, d_range):
    from paper_2602_05017_gb300 import binding
    rng = np.random.default_rng(shape[0] + 31 * shape[1])
    w = inputs.random_problem(rng, *shape, n_agents=200, dirichlet=True, D_range=d_range)
    if prec == "fp32":
        rho, start, bound = w.rho0.astype(np.float32), w.rho0, 1e-5
    else:
        t, start = rounded(w.rho0, prec)
        rho, bound = t.cuda(), 8 * UNIT_ROUNDOFF[prec] + 1e-5
    ref = oracle.Problem(**w.oracle_kwargs()).step(start, 2)
    sim = binding.BioFVM(w.nx, w.ny, w.nz, w.ns, w.dx, w.dt, w.D, w.lam, w.dirichlet_on,
                         w.dirichlet_value, precision=prec)
    assert sim.describe().split()[axis] == f"{'xyz'[axis]}=pipe/{tile}"
    sim.set_sources(w.voxel, w.secretion, w.target, w.uptake, w.weight)
    sim.set_density(rho)
    sim.step(2)
    got = as_f64(sim.density())
    sim.close()
    assert np.abs(got - ref).max() <= bound * np.abs(ref).max()
