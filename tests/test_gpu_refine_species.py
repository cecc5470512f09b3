"""GPU tests of the refined solve with fewer switching states than species: the
launches that the device turns into an exact gradient cover all species."""
import numpy as np
import pytest
import torch

import paper_2510_23739_gb300 as sw
from synth import Geometry, Switching

pytestmark = pytest.mark.gpu


def _problem(P, N, cycle, seed):
    g = Geometry(X=14, Y=11, Z=9, T=24, N=N, P=P, k=5, pulses_per_cycle=cycle)
    rng = np.random.default_rng(seed)
    s = Switching(tuple(rng.uniform(0.0, 0.2, P)), tuple(rng.uniform(0.5, 1.0, P)),
                  tuple(rng.uniform(0.0, 0.3, P)), 1.5)
    y = torch.tensor(rng.standard_normal(g.y_shape()), dtype=torch.float32, device="cuda")
    return g, s, rng.standard_normal(g.k_shape()), y


def _solve(op, y, prm):
    op.fista_init(y, prm)
    op.fista_step(6)
    return op.fista_get().clone()


# states: as many as the cycle has, one, and as few as there are pulses
@pytest.mark.parametrize("P,N,cycle", [(3, 6, 2), (3, 6, 1), (3, 1, 10), (8, 3, 2)])
@pytest.mark.parametrize("resync", ["fp32", "bf16x3", "bf16x6"])
def test_refined_solve_with_fewer_states_than_species(P, N, cycle, resync):
    """Alone by graph and by launches, and in a batch: equal to each other, and
    to the plain FP32 iterates to BF16's operator error (5e-3) in every species."""
    probs = [_problem(P, N, cycle, seed) for seed in range(2)]
    kw = dict(step=2e-4, lambda_l1=1e-2, lambda_tv=1e-2, inner_iters=4)
    prm = sw.SolveParams(**kw, refine_every=2, refine_precision=resync, refine_budget=0.05)
    ops = [sw.Operator(g, K, s) for g, s, K, _ in probs]
    try:
        want = [_solve(op, p[3], sw.SolveParams(**kw)) for op, p in zip(ops, probs)]
        for op in ops:
            op.set_precision("bf16")
        got = [_solve(op, p[3], prm) for op, p in zip(ops, probs)]
        for a, w in zip(got, want):
            assert (w.flatten(1).norm(dim=1) > 0).all()
            assert float(((a - w).flatten(1).norm(dim=1) / w.flatten(1).norm(dim=1)).max()) <= 5e-3
        for op, p in zip(ops, probs):
            op.fista_init(p[3], prm)
        b = sw.Batch(ops)
        b.step(6)
        for op, a in zip(ops, got):
            assert torch.equal(op.fista_get(), a)
        b.close()
        for op, p, a in zip(ops, probs, got):
            op.use_graphs(False)
            assert torch.equal(_solve(op, p[3], prm), a)
            op.check_device()
    finally:
        for op in ops:
            op.close()
