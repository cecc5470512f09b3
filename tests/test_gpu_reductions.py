"""GPU tests of the FP64 sums over long arrays (FP32 pairs in groups of 16)
at group tails, unaligned starts and value ranges, through the objective and
the parameter gradient.

Tolerance: the pairs drop less than 2^-43 of a group, FP64 sums of n terms
less than n 2^-53 (n <= 1e5 here): 1e-12 relative for sums of squares.
"""
import numpy as np
import pytest
import torch

import oracle
import paper_2510_23739_gb300 as sw
from synth import Geometry, Switching

pytestmark = pytest.mark.gpu


def _operator(X, Y, Z, T, N, seed=0):
    g = Geometry(X=X, Y=Y, Z=Z, T=T, N=N, P=2, k=3, pulses_per_cycle=2)
    s = Switching((0.1, 0.0), (1.0, 0.0), (0.0, 1.0), 2.0)
    K = np.random.default_rng(seed).standard_normal(g.k_shape())
    return g, s, K, sw.Operator(g, K, s)


@pytest.mark.parametrize("scale", [1.0, 1e-9, 1e-14, 1e-30, 1e18, 1e30])
@pytest.mark.parametrize("shape", [(1, 1, 2, 3, 1), (5, 7, 2, 511, 1), (16, 16, 2, 64, 2),
                                   (9, 11, 2, 77, 3)])
@pytest.mark.parametrize("shift", [0, 1])
def test_sum_of_squares_of_the_measurements(shape, scale, shift):
    g, s, K, op = _operator(*shape)
    try:
        y = (np.random.default_rng(1).standard_normal(g.y_shape()) * scale).astype(np.float32)
        buf = torch.zeros(y.size + shift, dtype=torch.float32, device="cuda")
        t = buf[shift:].view(*g.y_shape())
        t.copy_(torch.from_numpy(y))
        c = torch.zeros(g.c_shape(), dtype=torch.float32, device="cuda")
        F, fit = op.objective(c, t, 0.0, 0.0)
        want = 0.5 * float(np.sum(y.astype(np.float64) ** 2))
        assert abs(fit - want) <= 1e-12 * want
        t.view(-1)[-1] = np.inf
        assert not np.isfinite(op.objective(c, t, 0.0, 0.0)[1])
        t.view(-1)[-1] = np.nan
        assert np.isnan(op.objective(c, t, 0.0, 0.0)[1])
    finally:
        op.close()


@pytest.mark.parametrize("shape", [(1, 1, 3, 9, 2), (17, 16, 5, 12, 2), (40, 33, 131, 20, 2)])
def test_parameter_gradient_over_runs_of_positions(shape):
    """One position, a run and its tail, and more depths than a block's threads."""
    g, s, K, op = _operator(*shape, seed=2)
    try:
        rng = np.random.default_rng(3)
        c, w = rng.standard_normal(g.c_shape()), rng.standard_normal(g.y_shape())
        dk, dmu = op.param_vjp(torch.tensor(c, dtype=torch.float32, device="cuda"),
                               torch.tensor(w, dtype=torch.float32, device="cuda"))
        # <w, dH c> from the oracle's gradient of 1/2||H c - y||^2 with y = H c - w
        y = oracle.forward(g, s, K, c) - w
        want_k, want_mu = oracle.param_grad(g, s, K, c, y)
        scale = max(np.abs(want_k).max(), abs(want_mu))
        assert np.abs(dk - want_k).max() <= 1e-5 * scale
        assert abs(dmu - want_mu) <= 1e-5 * scale
    finally:
        op.close()
