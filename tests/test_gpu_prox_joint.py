"""GPU tests of the joint prox's first iterations (which read no dual, or one)
and of every species count, with states that fill and leave a group of four.

Tolerance (relative L2): clamped dual steps do not expand errors; each of up
to 3 iterations sums at most 11 states and 4 differences per voxel: 1e-5 as for
the other proximal maps.
"""
import numpy as np
import pytest
import torch

import oracle
import paper_2510_23739_gb300 as sw
from synth import Geometry, Switching

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("iters", [0, 1, 2, 3])
@pytest.mark.parametrize("P,Q,Y,X,Z", [(1, 1, 4, 5, 6), (2, 4, 1, 6, 9), (3, 5, 6, 1, 33),
                                       (4, 8, 3, 4, 1), (5, 3, 5, 4, 7), (6, 11, 4, 3, 5),
                                       (7, 2, 3, 5, 4), (8, 9, 7, 6, 13)])
def test_prox_joint_matches_oracle(P, Q, Y, X, Z, iters):
    g = Geometry(X=X, Y=Y, Z=Z, T=3, N=Q + 1, P=P, k=1, pulses_per_cycle=Q)
    rng = np.random.default_rng(P)
    s = Switching(tuple(rng.uniform(0, 0.3, P)), tuple(rng.uniform(0.5, 1, P)),
                  tuple(rng.uniform(0, 0.5, P)), 2.0)
    K = np.ones(g.k_shape())
    z = rng.standard_normal(g.c_shape()) + 0.3
    op = sw.Operator(g, K, s)
    try:
        lams = (0.3, 0.1, 0.2)
        step2 = 1.0 / op.prox_joint_step_bound(*lams)
        got = op.prox_joint(torch.tensor(z, dtype=torch.float32, device="cuda"), 0.6, *lams, iters,
                            step2).cpu().numpy()
        want = oracle.prox_joint(g, s, z, 0.6, *lams, iters, step2)
        assert np.linalg.norm(got - want) <= 1e-5 * np.linalg.norm(want)
    finally:
        op.close()
