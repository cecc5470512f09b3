"""GPU tests of the sums of products over long arrays: as accurate as sums in
FP64, through the data fit and the parameter gradient.

Tolerance: the reference (one correctly rounded addition of exact products,
math.fsum) against a thread's sums in FP64 and the trees over threads and
blocks: up to about 30 additions of 2^-53 relative to the sum of the products'
magnitudes, 3.3e-15.
"""
import math

import numpy as np
import pytest
import torch

import paper_2510_23739_gb300 as sw
from synth import Geometry, Switching

pytestmark = pytest.mark.gpu

TOL = 3.4e-15


def _values(kind, n, rng):
    if kind == "normal":
        return rng.standard_normal(n)
    if kind == "equal":  # roundings that all go the same way
        return np.full(n, 1.2345678)
    if kind == "wide":
        return rng.standard_normal(n) * 10.0 ** rng.integers(-9, 6, n)
    if kind == "sparse":  # exact zeros, and products below FP32's smallest
        return np.where(rng.random(n) < 0.1, rng.standard_normal(n), np.where(rng.random(n) < 0.1, 1e-30, 0))
    return rng.standard_normal(n) * 1e25  # products above FP32's largest


KINDS = ["normal", "equal", "wide", "sparse", "large"]


def _squares(v):
    return math.fsum((v.astype(np.float64) ** 2).tolist())


@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("shape", [(1, 1, 2, 16, 1), (4, 4, 2, 64, 1), (32, 33, 2, 128, 2),
                                   (65, 61, 2, 100, 4)])
def test_sum_of_squares_of_the_measurements(shape, kind):
    X, Y, Z, T, N = shape
    g = Geometry(X=X, Y=Y, Z=Z, T=T, N=N, P=2, k=3, pulses_per_cycle=2)
    s = Switching((0.1, 0.0), (1.0, 0.0), (0.0, 1.0), 2.0)
    op = sw.Operator(g, np.random.default_rng(0).standard_normal(g.k_shape()), s)
    try:
        y = _values(kind, int(np.prod(g.y_shape())), np.random.default_rng(1)).astype(np.float32)
        c = torch.zeros(g.c_shape(), dtype=torch.float32, device="cuda")
        fit = op.objective(c, torch.from_numpy(y).cuda().view(*g.y_shape()), 0.0, 0.0)[1]
        want = 0.5 * _squares(y)
        assert abs(fit - want) <= TOL * want
    finally:
        op.close()


@pytest.mark.parametrize("kind", ["normal", "equal", "wide", "sparse"])
@pytest.mark.parametrize("shape", [(3, 5, 2), (5, 7, 130), (48, 47, 3)])
def test_sums_of_the_parameter_gradient(shape, kind):
    """One species, no fluence decay and kappa = 0: the gradient in kappa is
    -sum g c with g = A^T w of the second pulse, which H^T w is too (the first
    pulse's w is zero)."""
    X, Y, Z = shape
    g = Geometry(X=X, Y=Y, Z=Z, T=9, N=2, P=1, k=3, pulses_per_cycle=2)
    s = Switching((0.0,), (1.0,), (0.0,), 0.0)
    rng = np.random.default_rng(2)
    K = rng.standard_normal(g.k_shape())
    c = _values(kind, int(np.prod(g.c_shape())), rng).astype(np.float32).reshape(g.c_shape())
    w = torch.zeros(g.y_shape(), device="cuda")
    w[1] = torch.tensor(rng.standard_normal(g.y_shape()[1:]), dtype=torch.float32)
    op = sw.Operator(g, K, s)
    try:
        prod = (op.adjoint(w).cpu().numpy().astype(np.float64) * c.astype(np.float64)).ravel()
        dk, _ = op.param_vjp(torch.from_numpy(c).cuda(), w)
        assert abs(dk[0] + math.fsum(prod.tolist())) <= TOL * math.fsum(np.abs(prod).tolist())
    finally:
        op.close()
