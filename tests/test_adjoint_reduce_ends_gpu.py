"""Infinities and NaN at the end of a line, where no difference follows, in the adjoint's parameter
sums (biofvm_param_grad_noalloc): the same infinities and NaN as numpy's sums."""
import numpy as np
import pytest

from test_adjoint_reduce_gpu import run, sums

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bad", [np.inf, -np.inf, np.nan])
@pytest.mark.parametrize("dtype", [np.float64, np.float32])
@pytest.mark.parametrize("shape", [(40, 33, 9, 2), (1, 7, 9, 2), (9, 1, 7, 3), (7, 9, 1, 1)],
                         ids=lambda s: "x".join(map(str, s)))
def test_line_ends(shape, dtype, bad):
    nx, ny, nz, ns = shape
    rng = np.random.default_rng(nx)
    mu, u = (rng.uniform(1.0, 2.0, (nz, ny, nx, ns)).astype(dtype) for _ in range(2))
    mu[-1, -1, -1, -1] = bad
    for axis in range(3):
        for got, want in zip(run(mu, u, axis), sums(mu, u, axis)):
            assert np.allclose(got, want, rtol=1e-12, equal_nan=True), (axis, got, want)
