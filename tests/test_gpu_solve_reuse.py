"""GPU tests of what a handle keeps between solves: iterations captured with
the same settings serve the next solve, others are captured again; and of the
backward pass that shares one A^T."""
import numpy as np
import pytest
import torch

import paper_2510_23739_gb300 as sw
from synth import Geometry, Switching

pytestmark = pytest.mark.gpu

GEOM = Geometry(X=14, Y=11, Z=9, T=24, N=6, P=2, k=5, pulses_per_cycle=3)
SW = Switching((0.1, 0.0), (1.0, 0.0), (0.05, 1.0), 2.0)
K = np.random.default_rng(0).standard_normal(GEOM.k_shape())


def _y(seed):
    return torch.tensor(np.random.default_rng(seed).standard_normal(GEOM.y_shape()),
                        dtype=torch.float32, device="cuda")


def _params(**kw):
    return sw.SolveParams(**{**dict(step=2e-4, lambda_l1=1e-2, lambda_tv=1e-2, inner_iters=4), **kw})


def _solve(op, y, prm):
    op.fista_init(y, prm)
    op.fista_step(5)
    return op.fista_get().clone()


@pytest.mark.parametrize("prec,kw", [("fp32", {}), ("bf16", sw.REFINED_DEFAULTS),
                                     ("bf16", dict(refine_every=2))])
def test_solves_of_one_handle_equal_those_of_fresh_handles(prec, kw):
    changes = [{}, {}, dict(step=1e-4), dict(step=1e-4), dict(lambda_tv=3e-2), dict(inner_iters=2),
               dict(momentum="none"), dict(lambda_3=1e-2), {}]
    one = sw.Operator(GEOM, K, SW, precision=prec)
    try:
        for i, ch in enumerate(changes):
            prm = _params(**{**kw, **ch})
            fresh = sw.Operator(GEOM, K, SW, precision=prec)
            want = _solve(fresh, _y(i), prm)
            fresh.close()
            assert torch.equal(_solve(one, _y(i), prm), want), ch
    finally:
        one.close()


@pytest.mark.parametrize("prec", ["fp32", "bf16x3", "bf16"])
@pytest.mark.parametrize("resync", ["fp32", "bf16x3", "bf16"])
@pytest.mark.parametrize("budget", [0.0, 0.05])
def test_resync_precisions(prec, resync, budget):
    """Every pair of increment and resync precisions, decided on the host or
    on the device: the plain FP32 iterates to BF16's operator error (5e-3)."""
    op = sw.Operator(GEOM, K, SW)
    try:
        want = _solve(op, _y(6), _params())
        op.set_precision(prec)
        got = _solve(op, _y(6), _params(refine_every=2, refine_precision=resync,
                                        refine_budget=budget))
        op.check_device()
        assert float((got - want).norm() / want.norm()) <= 5e-3
        if "bf16" not in (prec, resync):
            assert float((got - want).norm() / want.norm()) <= 1e-5
    finally:
        op.close()


def test_unpinning_a_tensor_core_schedule():
    """A schedule pinned before the precision is selected, then released."""
    op = sw.Operator(GEOM, K, SW)
    try:
        for kid in (0, 1):
            op.tc_schedule(kid, split=1)
        op.set_precision("bf16")
        c = torch.tensor(np.random.default_rng(7).standard_normal(GEOM.c_shape()),
                         dtype=torch.float32, device="cuda")
        pinned = op.forward(c), op.adjoint(_y(8))
        for kid in (0, 1):
            op.tc_schedule(kid)
        free = op.forward(c), op.adjoint(_y(8))
        op.check_device()
        for a, b in zip(pinned, free):
            assert float((a - b).norm() / b.norm()) <= 2e-5  # FP32 sums of the same products
    finally:
        op.close()


def test_a_restored_step_is_not_taken_for_the_next_solve():
    a, b = sw.Operator(GEOM, K, SW), sw.Operator(GEOM, K, SW)
    try:
        want = _solve(b, _y(1), _params())
        _solve(b, _y(1), _params(step=5e-5))
        state = b.fista_save()
        _solve(a, _y(1), _params())
        a.fista_restore(state)  # a step of 5e-5
        a.fista_step(2)
        assert torch.equal(_solve(a, _y(1), _params()), want)
    finally:
        a.close()
        b.close()


def test_batch_after_a_solve_with_other_settings():
    ops = [sw.Operator(GEOM, K, SW) for _ in range(2)]
    try:
        for op, prm in zip(ops, (_params(step=1e-4), _params())):
            _solve(op, _y(2), prm)
            op.fista_init(_y(3), _params())
        b = sw.Batch(ops)
        b.step(5)
        got = [op.fista_get().clone() for op in ops]
        b.close()
        want = _solve(ops[0], _y(3), _params())
        assert torch.equal(got[0], want) and torch.equal(got[1], want)
    finally:
        for op in ops:
            op.close()


@pytest.mark.parametrize("prec", ["fp32", "bf16", "fp8"])
def test_adjoint_vjp_is_adjoint_and_param_vjp(prec):
    op = sw.Operator(GEOM, K, SW, precision=prec)
    try:
        rng = np.random.default_rng(4)
        c = torch.tensor(rng.standard_normal(GEOM.c_shape()), dtype=torch.float32, device="cuda")
        gc, dk, dmu = op.adjoint_vjp(c, _y(5))
        want_k, want_mu = op.param_vjp(c, _y(5))
        assert np.array_equal(dk, want_k) and dmu == want_mu
        want = op.adjoint(_y(5))
        assert float((gc - want).norm() / want.norm()) <= 3e-6  # P^T before or after the transform
    finally:
        op.close()
