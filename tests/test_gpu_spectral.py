"""GPU tests of the spectral A and A^T (FFT over the scan plane) at the sizes
where they can go wrong, against the FP64 oracle.

Tolerance (relative L2): each of the two transforms per axis loses at most
about log2(L) roundings of 2^-24, L <= 256, and a product sums at most about
128 channels, whose roundings add up like sqrt(128): (4 x 8 + 11) 2^-24 = 2.6e-6.
"""
import numpy as np
import pytest
import torch

import oracle
import paper_2510_23739_gb300 as sw
from synth import Geometry, Switching

pytestmark = pytest.mark.gpu

TOL = 3e-6


def rel(a, b):
    return float(np.linalg.norm(a - b) / max(np.linalg.norm(b), 1e-300))


def dev(a):
    return torch.tensor(np.asarray(a), dtype=torch.float32, device="cuda")


def host(t):
    return t.detach().cpu().numpy().astype(np.float64)


def problem(X, Y, Z, T, N, P, k, cycle, seed=0, band=None):
    """Random kernel; band: samples reached per depth, moving with depth (None: all)."""
    g = Geometry(X=X, Y=Y, Z=Z, T=T, N=N, P=P, k=k, pulses_per_cycle=cycle)
    rng = np.random.default_rng(seed)
    s = Switching(tuple(rng.uniform(0.0, 0.2, P)), tuple(rng.uniform(0.5, 1.0, P)),
                  tuple(rng.uniform(0.0, 0.3, P)), 1.5)
    K = rng.standard_normal(g.k_shape())
    if band:
        t = np.arange(T)
        for j in range(Z):
            lo = j * max(1, T - band) // max(1, Z)
            K[j, :, :, (t < lo) | (t >= lo + band)] = 0.0
    return g, s, K


# one tile at a length's limit and just past it, several tiles along either
# axis and both, more states than a block takes, more species than four, odd
# and single channels, bands whose groups are empty or partial, and supports
# as wide as the scan
SHAPES = {
    "at_length": dict(X=14, Y=18, Z=6, T=20, N=3, P=2, k=5, cycle=3),
    "past_length": dict(X=15, Y=19, Z=6, T=20, N=3, P=2, k=5, cycle=3),
    "tiles_x": dict(X=270, Y=3, Z=3, T=9, N=2, P=2, k=5, cycle=2),
    "tiles_y": dict(X=2, Y=301, Z=2, T=7, N=2, P=1, k=3, cycle=2),
    "tiles_both": dict(X=259, Y=257, Z=1, T=3, N=1, P=1, k=3, cycle=1),
    "states_23": dict(X=9, Y=7, Z=5, T=11, N=25, P=2, k=3, cycle=23),
    "states_13_species_6": dict(X=7, Y=9, Z=9, T=17, N=13, P=6, k=3, cycle=13),
    "one_depth": dict(X=11, Y=6, Z=1, T=13, N=2, P=1, k=7, cycle=2),
    "one_sample": dict(X=11, Y=6, Z=5, T=1, N=2, P=2, k=3, cycle=2),
    "band": dict(X=10, Y=12, Z=33, T=75, N=4, P=3, k=5, cycle=2, band=6),
    "band_wide": dict(X=10, Y=12, Z=19, T=41, N=4, P=2, k=5, cycle=4, band=23),
    "support_63": dict(X=5, Y=4, Z=3, T=10, N=1, P=1, k=63, cycle=1),
}


@pytest.mark.parametrize("name", list(SHAPES))
def test_operator_matches_oracle(name):
    g, s, K = problem(**SHAPES[name])
    rng = np.random.default_rng(1)
    c, y = rng.standard_normal(g.c_shape()), rng.standard_normal(g.y_shape())
    op = sw.Operator(g, K, s)
    try:
        assert rel(host(op.forward(dev(c))), oracle.forward(g, s, K, c)) <= TOL
        assert rel(host(op.adjoint(dev(y))), oracle.adjoint(g, s, K, y)) <= TOL
    finally:
        op.close()


@pytest.mark.parametrize("name", ["at_length", "tiles_x", "states_13_species_6", "band"])
def test_gradient_matches_oracle(name):
    """The gradient (A, residual and A^T without u in between, or tile by
    tile) per state, through one plain iteration without the prox."""
    g, s, K = problem(**SHAPES[name])
    y = np.random.default_rng(2).standard_normal(g.y_shape())
    op = sw.Operator(g, K, s)
    try:
        op.fista_init(dev(y), sw.SolveParams(step=1e-3, lambda_l1=0.0, lambda_tv=0.0))
        op.fista_step(3)
        want = oracle.fista(g, s, K, y, 1e-3, 3, 0.0, 0.0, 0)
        assert rel(host(op.fista_get()), want) <= 10 * TOL  # three gradients
    finally:
        op.close()


@pytest.mark.parametrize("name", ["at_length", "tiles_x", "states_23", "band"])
def test_unaligned_arrays(name):
    """Inputs and outputs that start 4 bytes past an aligned address."""
    g, s, K = problem(**SHAPES[name])
    rng = np.random.default_rng(3)
    c, y = rng.standard_normal(g.c_shape()), rng.standard_normal(g.y_shape())
    op = sw.Operator(g, K, s)

    def shifted(shape, value=None):
        n = int(np.prod(shape))
        t = torch.zeros(n + 1, dtype=torch.float32, device="cuda")[1:].view(*shape)
        if value is not None:
            t.copy_(dev(value))
        return t

    try:
        a, b = shifted(g.c_shape(), c), shifted(g.y_shape(), y)
        f = op.forward(a, out=shifted(g.y_shape()))
        assert torch.equal(f, op.forward(dev(c)))
        assert torch.equal(op.adjoint(b, out=shifted(g.c_shape())), op.adjoint(dev(y)))
    finally:
        op.close()


@pytest.mark.parametrize("name", ["at_length", "tiles_x", "band"])
def test_bf16_rounds_as_the_tensor_core_kernels_do(name):
    """BF16 operands: the spectral kernels and the tensor-core ones (pinned)
    round the same values, so they differ by FP32 sums only (a few hundred
    accumulations of 2^-24)."""
    g, s, K = problem(**SHAPES[name])
    rng = np.random.default_rng(4)
    c, y = dev(rng.standard_normal(g.c_shape())), dev(rng.standard_normal(g.y_shape()))
    op = sw.Operator(g, K, s, precision="bf16")
    try:
        f, a = op.forward(c), op.adjoint(y)
        for kid in (0, 1):
            op.tc_schedule(kid, split=1)
        ft, at = op.forward(c), op.adjoint(y)
        assert not torch.equal(a, at)  # another kernel ran
        assert rel(host(f), host(ft)) <= 2e-5
        assert rel(host(a), host(at)) <= 2e-5
    finally:
        op.close()


@pytest.mark.parametrize("value", [np.inf, np.nan])
@pytest.mark.parametrize("name", ["at_length", "tiles_x", "band"])
def test_non_finite_inputs_stay_within_their_support(name, value):
    """An infinity or NaN reaches the outputs whose sums hold it and no others."""
    g, s, K = problem(**SHAPES[name])
    r = g.k // 2
    rng = np.random.default_rng(5)
    c, y = rng.standard_normal(g.c_shape()), rng.standard_normal(g.y_shape())
    py, px, pj, pt = g.Y // 2, g.X // 3, g.Z // 2, int(np.flatnonzero(K[g.Z // 2].any((0, 1)))[1])
    op = sw.Operator(g, K, s)
    try:
        ref_f, ref_a = oracle.forward(g, s, K, c), oracle.adjoint(g, s, K, y)
        c[0, py, px, pj] = value
        y[0, py, px, pt] = value
        got_f, got_a = host(op.forward(dev(c))), host(op.adjoint(dev(y)))
        near = np.zeros((g.Y, g.X), dtype=bool)
        near[max(0, py - r):py + r + 1, max(0, px - r):px + r + 1] = True
        assert np.isfinite(got_f[:, ~near]).all() and np.isfinite(got_a[:, ~near]).all()
        assert rel(got_f[:, ~near], ref_f[:, ~near]) <= 1e-5
        assert rel(got_a[:, ~near], ref_a[:, ~near]) <= 1e-5
        hit = K[pj, r, r] != 0  # the sample's own tap, at its own position
        assert not np.isfinite(got_f[:, py, px][:, hit]).any()
        assert not np.isfinite(got_a[:, py, px][:, K[:, r, r, pt] != 0]).any()
    finally:
        op.close()


def test_solve_with_a_nan_measurement_keeps_the_rest():
    """A dead pixel (NaN) blanks its neighbourhood of the solution only, as
    the l1 and nonnegativity step maps NaN to 0."""
    g, s, K = problem(X=24, Y=20, Z=4, T=12, N=3, P=2, k=3, cycle=3)
    y = np.random.default_rng(6).standard_normal(g.y_shape())
    prm = sw.SolveParams(step=2e-3, lambda_l1=1e-3, lambda_tv=0.0)
    op = sw.Operator(g, K, s)
    try:
        op.fista_init(dev(y), prm)
        op.fista_step(1)
        whole = op.fista_get().clone()
        y[1, 10, 12, :] = np.nan
        op.fista_init(dev(y), prm)
        op.fista_step(1)
        got = op.fista_get()
        near = torch.zeros(g.Y, g.X, dtype=torch.bool, device="cuda")
        near[9:12, 11:14] = True
        assert torch.isfinite(got).all()
        assert (got[:, near] == 0).all()
        assert float((got - whole)[:, ~near].norm() / whole[:, ~near].norm()) <= 1e-5
    finally:
        op.close()


@pytest.mark.parametrize("X,Y", [(16, 18), (11, 258), (257, 5)])
def test_one_tap(X, Y):
    """k = 1: tiles that do not overlap, one where the scan fits, else several."""
    g, s, K = problem(X=X, Y=Y, Z=5, T=12, N=3, P=2, k=1, cycle=2)
    rng = np.random.default_rng(9)
    c, y = rng.standard_normal(g.c_shape()), rng.standard_normal(g.y_shape())
    op = sw.Operator(g, K, s)
    try:
        assert rel(host(op.forward(dev(c))), oracle.forward(g, s, K, c)) <= TOL
        assert rel(host(op.adjoint(dev(y))), oracle.adjoint(g, s, K, y)) <= TOL
    finally:
        op.close()
