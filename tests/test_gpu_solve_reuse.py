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
