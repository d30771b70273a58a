"""The adjoint's parameter sums of FP32 fields keep FP64's precision: against exact sums
(rationals; quadruple precision where numpy's long double has it), with magnitudes that meet and
that never meet in one element.

Bound: a sum's terms pass at most k roundings to 53 bits -- 16 for a group of eight added in FP64,
8 in the block's tree, 16 + 5 over the blocks of the final sum -- so k 2^-53 of the sum of the
terms' sizes, k = 45; k = 16 where one group is the whole sum (pairs of floats, 48 bits, leave up to
8 x 2^-48 there).
"""
from fractions import Fraction

import numpy as np
import pytest

from test_adjoint_reduce_gpu import run

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("decay", [0, 3, 7, 9, 12, 20])
def test_one_group(decay):
    """32 sums of eight elements each: mu falls by 2^decay an element where u rises by it."""
    rng = np.random.default_rng(decay)
    i = np.arange(8)[None, :, None, None]
    worst = 0
    for rise in (decay * (i - 7), -decay * i):  # against each other, then together
        mu = (rng.normal(size=(1, 8, 1, 32)) * 2.0 ** (-decay * i)).astype(np.float32)
        u = (rng.normal(size=(1, 8, 1, 32)) * 2.0 ** rise).astype(np.float32)
        for got, terms in zip(run(mu, u, 1), (lambda m, v: [x * y for x, y in zip(m, v)],
                                              lambda m, v: [(m[k + 1] - m[k]) * (v[k + 1] - v[k])
                                                            for k in range(7)])):
            for s in range(32):
                t = terms(*([Fraction(float(x)) for x in a[0, :, 0, s]] for a in (mu, u)))
                err = abs(Fraction(float(got[s])) - sum(t)) / sum(map(abs, t))
                assert err <= 16 * Fraction(1, 2 ** 53), (s, float(err))
                worst = max(worst, float(err))
    print(f"decay {decay}: {worst:.2e} of the sum of sizes")


@pytest.mark.skipif(np.finfo(np.longdouble).nmant < 100, reason="needs quadruple precision")
@pytest.mark.parametrize("scale", [0.05, 0.5, 1.2])
def test_disjoint_peaks(scale):
    """mu and u peak in opposite corners and fall by 2^-scale a voxel in every direction."""
    nz, ny, nx = 64, 96, 192
    rng = np.random.default_rng(5)
    z, y, x = np.meshgrid(np.arange(nz), np.arange(ny), np.arange(nx), indexing="ij")
    near, far = x + y + z, (nx - 1 - x) + (ny - 1 - y) + (nz - 1 - z)
    mu, u = ((rng.uniform(0.5, 1.0, near.shape) * 2.0 ** (-scale * dist))
             .astype(np.float32)[..., None] for dist in (near, far))
    q_mu, q_u = mu.astype(np.longdouble), u.astype(np.longdouble)
    for axis in range(3):
        d_mu, d_u = np.diff(q_mu, axis=2 - axis), np.diff(q_u, axis=2 - axis)
        for got, t in zip(run(mu, u, axis), (q_mu * q_u, d_mu * d_u)):
            assert abs(got[0] - t.sum()) <= 45 * 2.0 ** -53 * abs(t).sum(), (axis, got[0])
