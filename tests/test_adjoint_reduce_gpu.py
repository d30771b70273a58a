"""The adjoint's parameter-gradient sums on their own (biofvm_param_grad_noalloc), against the
same sums in numpy at 64 bits: lines around one and several segments of 32 positions, one voxel,
substrate counts that do and do not divide a block, zeros, subnormals and infinities.

Bound: FP64 sums, or floats eight at a time to no fewer bits: the result lies within (terms per sum)
x 2^-53 of the sum of the terms' sizes, which 1e-13 covers (test_adjoint_reduce_bits_gpu.py holds
them closer).
"""
import ctypes

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def sums(mu, u, axis):
    mu, u = mu.astype(np.float64), u.astype(np.float64)
    dm, du = np.diff(mu, axis=2 - axis), np.diff(u, axis=2 - axis)
    red = lambda t: t.reshape(-1, t.shape[3]).sum(0)
    return red(mu * u), red(dm * du), red(abs(mu * u)), red(abs(dm * du))


def run(mu, u, axis, nan=False):
    import torch
    from paper_2602_05017_gb300 import binding
    lib = binding.load()
    nz, ny, nx, ns = mu.shape
    code = binding.FP64 if mu.dtype == np.float64 else binding.FP32
    tm, tu = torch.tensor(mu, device="cuda"), torch.tensor(u, device="cuda")
    dD, dl = (torch.zeros(ns, dtype=torch.float64, device="cuda") for _ in range(2))
    st = lib.biofvm_param_grad_noalloc(
        ctypes.c_void_p(tm.data_ptr()), ctypes.c_void_p(tu.data_ptr()), nx, ny, nz, ns, axis, code,
        3.0, 1.0, ctypes.c_void_p(dD.data_ptr()), ctypes.c_void_p(dl.data_ptr()),
        torch.cuda.current_stream().cuda_stream)  # dt = 3, h = 1: -1 and -3 times the sums
    assert st == binding.OK
    torch.cuda.synchronize()
    return -dl.cpu().numpy(), -dD.cpu().numpy() / 3.0


@pytest.mark.parametrize("dtype", [np.float64, np.float32])
@pytest.mark.parametrize("shape", [(1, 1, 1, 1), (33, 32, 31, 1), (7, 65, 3, 3), (64, 2, 97, 5),
                                   (40, 9, 11, 32), (1, 200, 70, 2)],
                         ids=lambda s: "x".join(map(str, s)))
def test_sums_match_numpy(shape, dtype):
    nx, ny, nz, ns = shape
    rng = np.random.default_rng(nx + ny)
    mu = (rng.normal(size=(nz, ny, nx, ns)) * 2.0 ** rng.integers(-20, 20, (nz, ny, nx, ns)))
    mu[rng.random(mu.shape) < 0.3] = 0.0
    mu, u = mu.astype(dtype), rng.uniform(-3.0, 38.0, (nz, ny, nx, ns)).astype(dtype)
    for axis in range(3):
        s1, s2, a1, a2 = sums(mu, u, axis)
        g1, g2 = run(mu, u, axis)
        assert (abs(g1 - s1) <= 1e-13 * a1).all() and (abs(g2 - s2) <= 1e-13 * a2).all()


def test_subnormal_and_infinite_floats():
    rng = np.random.default_rng(3)
    mu = (rng.normal(size=(5, 6, 40, 2)) * 2.0 ** rng.uniform(-148, -120, (5, 6, 40, 2)))
    mu, u = mu.astype(np.float32), rng.uniform(1.0, 38.0, (5, 6, 40, 2)).astype(np.float32)
    for axis in range(3):
        s1, s2, a1, a2 = sums(mu, u, axis)
        g1, g2 = run(mu, u, axis)
        assert (abs(g1 - s1) <= 1e-13 * a1).all() and (abs(g2 - s2) <= 1e-13 * a2).all()
    mu[2, 3, 7, 1] = np.inf
    for axis in range(3):
        g1, _ = run(mu, u, axis)
        assert np.isfinite(g1[0]) and g1[1] == np.inf
