"""GPU tests of the on-chip TV prox at the edges of its tiles, warps and
rounds, against the FP64 oracle.

Tolerance: the clamped dual steps do not expand errors; each of up to 70
iterations adds a few roundings of 2^-24: 70 x 4 x 2^-24 = 1.7e-5 worst, and
they are not all one way: 1e-5 relative L2.
"""
import numpy as np
import pytest
import torch

import oracle
import paper_2510_23739_gb300 as sw
from synth import Geometry, Switching

pytestmark = pytest.mark.gpu


def _operator(P, Y, X, Z):
    g = Geometry(X=X, Y=Y, Z=Z, T=4, N=1, P=P, k=1, pulses_per_cycle=1)
    s = Switching((0.0,) * P, (0.0,) * P, (1.0,) * P, 0.0)
    K = np.zeros(g.k_shape())
    K[..., 0] = 1.0
    return sw.Operator(g, K, s)


# (P, Y, X, Z): depths at and around the lanes' 32, 64, 96 and 128; scans that
# leave partial tiles, one row, one column; volumes whose species take turns
SHAPES = [(1, 1, 1, 1), (2, 3, 5, 31), (1, 7, 9, 32), (2, 9, 7, 33), (1, 13, 6, 64), (2, 6, 13, 65),
          (1, 5, 11, 96), (2, 11, 5, 97), (1, 4, 9, 128), (3, 1, 70, 20), (3, 70, 1, 20),
          (2, 127, 97, 70), (3, 101, 90, 95), (2, 77, 83, 127)]


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("iters", [1, 2, 7])
def test_prox_tv_matches_oracle(shape, iters):
    op = _operator(*shape)
    try:
        z = np.random.default_rng(sum(shape)).standard_normal(shape)
        got = op.prox_tv(torch.tensor(z, dtype=torch.float32, device="cuda"), 0.2, iters)
        op.check_device()
        want = oracle.prox_tv(z, 0.2, iters)
        err = np.linalg.norm(got.cpu().numpy() - want) / np.linalg.norm(want)
        assert err <= 1e-5
    finally:
        op.close()


@pytest.mark.parametrize("momentum", ["beck_teboulle", "paper_printed", "none"])
def test_more_iterations_than_the_coefficient_table(momentum):
    op = _operator(2, 9, 10, 40)
    try:
        z = np.random.default_rng(1).standard_normal((2, 9, 10, 40))
        zt = torch.tensor(z, dtype=torch.float32, device="cuda")
        for iters in (64, 65, 70):
            got = op.prox_tv(zt, 0.3, iters, momentum=momentum).cpu().numpy()
            want = oracle.prox_tv(z, 0.3, iters, momentum=momentum)
            assert np.linalg.norm(got - want) / np.linalg.norm(want) <= 1e-5
    finally:
        op.close()


@pytest.mark.parametrize("value", [np.inf, -np.inf, np.nan])
@pytest.mark.parametrize("at", [(0, 0, 0, 0), (0, 8, 10, 39), (1, 4, 5, 31), (0, 3, 10, 32)])
def test_non_finite_entries_reach_their_neighbours_only(value, at):
    """Two iterations: entries more than three steps away see nothing of it (a
    dual entry is clamped to tau whatever it was)."""
    op = _operator(2, 9, 11, 40)
    try:
        z = np.random.default_rng(2).standard_normal((2, 9, 11, 40)).astype(np.float32)
        ref = op.prox_tv(torch.tensor(z, device="cuda"), 0.2, 2).cpu().numpy()
        z[at] = value
        got = op.prox_tv(torch.tensor(z, device="cuda"), 0.2, 2).cpu().numpy()
        far = np.sum([np.abs(i - c) for i, c in zip(np.indices(z.shape)[1:], at[1:])], axis=0) > 3
        far |= np.indices(z.shape)[0] != at[0]
        assert np.array_equal(got[far], ref[far])
        assert not np.isfinite(got[at])
        assert np.isfinite(np.delete(got.ravel(), np.ravel_multi_index(at, z.shape))).all()
    finally:
        op.close()
