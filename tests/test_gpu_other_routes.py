"""GPU tests of the kernels that serve what the transforms do not: the
tensor-core contractions (with a pinned schedule), the direct FP32 sums (a time
window that the product of the spectra cannot stage), and the refined solve on
scans of several tiles, each against the FP64 oracle or the plain FP32 iterates.

Tolerances (relative L2), from the arithmetic: two-term BF16 keeps each product
to 3 2^-16 (4e-5 of a sum), three terms to FP32's own (1e-5), BF16 rounds both
operands by up to 2^-8 (5e-3); FP32 sums of up to 10^4 terms, 1e-5.
"""
import numpy as np
import pytest
import torch

import oracle
import paper_2510_23739_gb300 as sw
from synth import Geometry, Switching

pytestmark = pytest.mark.gpu

TC_TOL = {"bf16x6": 1e-5, "bf16x3": 4e-5, "bf16": 5e-3}
SW2 = Switching((0.1, 0.0), (1.0, 0.0), (0.0, 1.0), 2.0)
SW3 = Switching((0.04, 0.09, 0.0), (1.0, 0.8, 0.0), (0.0, 0.1, 1.0), 3.0)
SHAPES = {
    "even": (dict(X=16, Y=16, Z=24, T=64, N=8, P=2, k=7, pulses_per_cycle=8), SW2),
    "ragged": (dict(X=13, Y=11, Z=37, T=57, N=7, P=3, k=5, pulses_per_cycle=3), SW3),
    "one_tap": (dict(X=17, Y=5, Z=3, T=20, N=1, P=1, k=1, pulses_per_cycle=5),
                Switching((0.0,), (0.0,), (1.0,), 0.0)),
    "one_column": (dict(X=1, Y=1, Z=5, T=33, N=4, P=2, k=3, pulses_per_cycle=2), SW2),
    "wide_support": (dict(X=12, Y=10, Z=24, T=80, N=3, P=2, k=11, pulses_per_cycle=3), SW2),
}
# more samples in the window than two states' images of the product leave room for
# (1376 with 57 depths or more, 1712 with up to 8)
LONG = {
    "long": (dict(X=9, Y=7, Z=5, T=1800, N=5, P=2, k=3, pulses_per_cycle=3), SW2),
    "long_ragged": (dict(X=35, Y=3, Z=9, T=1711, N=2, P=3, k=5, pulses_per_cycle=4), SW3),
}


def rel(a, b):
    return float(np.linalg.norm(a - b) / max(np.linalg.norm(b), 1e-300))


def dev(a):
    return torch.tensor(np.asarray(a), dtype=torch.float32, device="cuda")


def host(t):
    return t.detach().cpu().numpy().astype(np.float64)


def problem(shape, seed=0):
    g, s = Geometry(**shape[0]), shape[1]
    return g, s, np.random.default_rng(seed).standard_normal(g.k_shape())


def launches(op, f):
    before = op.launch_count()
    f()
    return op.launch_count() - before


def pin(op):
    for kernel in (0, 1):
        op.tc_schedule(kernel, split=1)


@pytest.mark.parametrize("prec", list(TC_TOL))
@pytest.mark.parametrize("name", list(SHAPES))
def test_pinned_tensor_core_operator_matches_oracle(name, prec):
    g, s, K = problem(SHAPES[name])
    rng = np.random.default_rng(30)
    c, y = rng.standard_normal(g.c_shape()), rng.standard_normal(g.y_shape())
    op = sw.Operator(g, K, s)
    try:
        pin(op)
        op.set_precision(prec)
        op.tc_schedule_info(0)
        f, a = op.forward(dev(c)), op.adjoint(dev(y))
        assert launches(op, lambda: op.forward(dev(c))) == 3  # states, contraction, rows of y
        assert torch.equal(op.forward(dev(c)), f) and torch.equal(op.adjoint(dev(y)), a)
        op.check_device()
        assert rel(host(f), oracle.forward(g, s, K, c)) <= TC_TOL[prec]
        assert rel(host(a), oracle.adjoint(g, s, K, y)) <= TC_TOL[prec]
    finally:
        op.close()


@pytest.mark.parametrize("prec,kw", [("bf16x3", dict()), ("bf16x6", dict()),
                                     ("bf16", dict(refine_every=2, refine_budget=0.05))])
def test_pinned_tensor_core_solve_and_gradients_match_oracle(prec, kw):
    g, s, K = problem(SHAPES["ragged"])
    rng = np.random.default_rng(31)
    y = rng.standard_normal(g.y_shape())
    op = sw.Operator(g, K, s)
    try:
        pin(op)
        op.set_precision(prec)
        v0 = rng.standard_normal(g.c_shape())
        L = op.lipschitz(30, dev(v0))
        assert L == pytest.approx(oracle.power(g, s, K, v0, 30), rel=5e-3 if prec == "bf16" else 1e-4)
        step = 0.9 / L
        op.fista_init(dev(y), sw.SolveParams(step=step, lambda_l1=0.01, lambda_tv=0.01, inner_iters=4,
                                             **kw))
        op.fista_step(8)
        op.check_device()
        want = oracle.fista(g, s, K, y, step, 8, 0.01, 0.01, 4)
        assert rel(host(op.fista_get()), want) <= (1e-3 if prec == "bf16" else 1e-4)
        if prec != "bf16":
            c = np.abs(rng.standard_normal(g.c_shape()))
            dk, dmu = op.param_grad(dev(c), dev(y))
            wk, wmu = oracle.param_grad(g, s, K, c, y)
            scale = max(np.abs(wk).max(), abs(wmu))
            assert np.abs(dk - wk).max() <= 1e-4 * scale and abs(dmu - wmu) <= 1e-4 * scale
    finally:
        op.close()


@pytest.mark.parametrize("name", list(LONG))
def test_direct_kernels_match_oracle(name):
    g, s, K = problem(LONG[name])
    rng = np.random.default_rng(32)
    c, y = rng.standard_normal(g.c_shape()), rng.standard_normal(g.y_shape())
    op = sw.Operator(g, K, s)
    try:
        assert launches(op, lambda: op.forward(dev(c))) == 3  # states, contraction, rows of y
        assert rel(host(op.forward(dev(c))), oracle.forward(g, s, K, c)) <= 1e-5
        assert rel(host(op.adjoint(dev(y))), oracle.adjoint(g, s, K, y)) <= 1e-5
        step = 0.9 / oracle.power(g, s, K, rng.standard_normal(g.c_shape()), 50)
        got, stats = op.solve(dev(y), sw.SolveParams(step=step, max_iters=6, lambda_l1=0.01,
                                                     lambda_tv=0.01, inner_iters=4))
        want = oracle.fista(g, s, K, y, step, 6, 0.01, 0.01, 4)
        assert rel(host(got), want) <= 1e-4
        F, fit = oracle.objective(g, s, K, want, y, 0.01, 0.01)
        assert stats["objective"] == pytest.approx(F, rel=1e-4)
        a = np.abs(c)
        dk, dmu = op.param_grad(dev(a), dev(y))
        wk, wmu = oracle.param_grad(g, s, K, a, y)
        scale = max(np.abs(wk).max(), abs(wmu))
        assert np.abs(dk - wk).max() <= 1e-4 * scale and abs(dmu - wmu) <= 1e-4 * scale
        # no tensor-core kernel takes so long a window
        with pytest.raises(sw.SwoptError, match="time window"):
            op.set_precision("bf16")
        assert launches(op, lambda: op.forward(dev(c))) == 3
    finally:
        op.close()


def test_direct_kernels_keep_infinities_local():
    g, s, K = problem(LONG["long_ragged"])
    rng = np.random.default_rng(33)
    c = rng.standard_normal(g.c_shape())
    op = sw.Operator(g, K, s)
    try:
        want = host(op.forward(dev(c)))
        c[0, 1, 17, 3] = np.inf
        got = host(op.forward(dev(c)))
        near = np.zeros((g.Y, g.X), dtype=bool)
        near[:, 15:20] = True
        assert np.array_equal(got[:, ~near], want[:, ~near])
        assert not np.isfinite(got[:, 1, 17]).any()
    finally:
        op.close()


@pytest.mark.parametrize("kw", [dict(refine_every=2), dict(refine_every=2, refine_budget=0.05)])
@pytest.mark.parametrize("prec,resync,tol", [("bf16", "bf16x3", 5e-3), ("bf16", "fp32", 5e-3),
                                             ("bf16x3", "fp32", 1e-5), ("fp32", "fp32", 1e-5)])
@pytest.mark.parametrize("P,cycle", [(2, 2), (3, 1)])
def test_refined_solve_on_several_tiles(kw, prec, resync, tol, P, cycle):
    """A scan wider than the largest transform: both branches of the schedule
    behind the gate, or the host's choice between them."""
    g = Geometry(X=270, Y=6, Z=4, T=9, N=2, P=P, k=5, pulses_per_cycle=cycle)
    s = SW2 if P == 2 else SW3
    rng = np.random.default_rng(34)
    K, y = rng.standard_normal(g.k_shape()), dev(rng.standard_normal(g.y_shape()))
    base = dict(step=5e-4, lambda_l1=1e-2, lambda_tv=1e-2, inner_iters=4)
    op = sw.Operator(g, K, s)
    try:
        op.fista_init(y, sw.SolveParams(**base))
        op.fista_step(6)
        want = host(op.fista_get())
        op.set_precision(prec)
        op.fista_init(y, sw.SolveParams(**base, refine_precision=resync, **kw))
        op.fista_step(6)
        op.check_device()
        got = host(op.fista_get())
        for p in range(P):
            assert rel(got[p], want[p]) <= tol
    finally:
        op.close()


@pytest.mark.parametrize("prec,refine,budget", [("bf16", 3, 0.0), ("bf16", 25, 0.1), ("bf16x3", 0, 0.0)])
def test_batch_by_transforms_matches_oracle(prec, refine, budget):
    ops, refs, ys, prms = [], [], [], []
    try:
        for i, name in enumerate(["even", "ragged", "wide_support"]):
            g, s, K = problem(SHAPES[name], seed=i)
            op = sw.Operator(g, K, s, precision=prec)
            ops.append(op)
            y = np.random.default_rng(70 + i).standard_normal(g.y_shape())
            step = 0.9 / oracle.power(g, s, K, np.random.default_rng(5).standard_normal(g.c_shape()), 50)
            prms.append(sw.SolveParams(step=step, lambda_l1=0.01, lambda_tv=0.01, inner_iters=4,
                                       refine_every=refine, refine_precision="bf16x3",
                                       refine_budget=budget))
            ys.append(dev(y))
            op.fista_init(ys[-1], prms[-1])
            refs.append(oracle.fista(g, s, K, y, step, 9, 0.01, 0.01, 4))
        b = sw.Batch(ops)
        b.step(9)
        assert not b.shared_in_use()
        got = [op.fista_get().clone() for op in ops]
        b.close()
        # as for the solves alone: BF16 increments between fixed resyncs leave 1e-3
        tol = 1e-3 if prec == "bf16" and budget == 0.0 else 1e-4
        for op, c, ref, y, prm in zip(ops, got, refs, ys, prms):
            op.check_device()
            assert rel(host(c), ref) <= tol
            op.fista_init(y, prm)
            op.fista_step(9)
            assert torch.equal(op.fista_get(), c)
    finally:
        for op in ops:
            op.close()
