"""GPU tests of pulse trains that never complete their cycle: any
pulses_per_cycle >= N is the same train, up to the largest int."""
import dataclasses

import numpy as np
import pytest
import torch

import paper_2510_23739_gb300 as sw
from synth import Geometry, Switching

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T", [24, 23])  # rows of y by 16-byte and by 4-byte accesses
@pytest.mark.parametrize("prec", ["fp32", "bf16"])
@pytest.mark.parametrize("cycle", [4, 2**31 - 3, 2**31 - 1])
def test_cycles_past_the_last_pulse(cycle, prec, T):
    g = Geometry(X=14, Y=11, Z=9, T=T, N=3, P=2, k=5, pulses_per_cycle=3)
    s = Switching((0.1, 0.0), (1.0, 0.0), (0.05, 1.0), 2.0)
    rng = np.random.default_rng(0)
    K = rng.standard_normal(g.k_shape())
    c = torch.tensor(rng.standard_normal(g.c_shape()), dtype=torch.float32, device="cuda")
    y = torch.tensor(rng.standard_normal(g.y_shape()), dtype=torch.float32, device="cuda")
    prm = sw.SolveParams(step=2e-4, lambda_l1=1e-2, lambda_tv=1e-2, inner_iters=3, max_iters=3)
    out = []
    for geom in (g, dataclasses.replace(g, pulses_per_cycle=cycle)):
        op = sw.Operator(geom, K, s, precision=prec)
        x, stats = op.solve(y, prm)
        out.append((op.forward(c), op.adjoint(y), x, stats["objective"], op.param_grad(c, y)))
        op.check_device()
        op.close()
    for a, b in zip(out[0][:3], out[1][:3]):
        assert torch.equal(a, b)
    assert out[0][3] == out[1][3]
    assert np.array_equal(out[0][4][0], out[1][4][0]) and out[0][4][1] == out[1][4][1]
