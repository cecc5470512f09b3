"""GPU tests of infinities, NaNs and masks of a huge value in the inputs of the
spectral operators: they reach the outputs whose sums contain them and no
others, in single calls and in solves, and cost what they touch.

Tolerances: away from the values, those of clean inputs (tests of the spectral
operators: 3e-6 in the norm); next to a huge value v, the sums are v K plus what
is 1e-29 of it: FP32 roundings of one product and of P^T's few terms, 1e-6."""
import numpy as np
import pytest
import torch

import oracle
import paper_2510_23739_gb300 as sw
from synth import Geometry, Switching

pytestmark = pytest.mark.gpu

# one tile, several tiles, and fewer states than species
SHAPES = {
    "one_tile": dict(X=41, Y=38, Z=9, T=23, N=6, P=2, k=5, cycle=3),
    "tiles": dict(X=270, Y=11, Z=3, T=9, N=2, P=2, k=5, cycle=2),
    "species": dict(X=30, Y=33, Z=6, T=20, N=3, P=3, k=3, cycle=1),
}
TOL = 3e-6


def rel(a, b):
    return float(np.linalg.norm(a - b) / max(np.linalg.norm(b), 1e-300))


def dev(a):
    return torch.tensor(np.asarray(a), dtype=torch.float32, device="cuda")


def host(t):
    return t.detach().cpu().numpy().astype(np.float64)


def problem(X, Y, Z, T, N, P, k, cycle, seed=0):
    g = Geometry(X=X, Y=Y, Z=Z, T=T, N=N, P=P, k=k, pulses_per_cycle=cycle)
    rng = np.random.default_rng(seed)
    s = Switching(tuple(rng.uniform(0.0, 0.2, P)), tuple(rng.uniform(0.5, 1.0, P)),
                  tuple(rng.uniform(0.1, 0.3, P)), 1.5)
    return g, s, rng.standard_normal(g.k_shape())


def near(g, points, reach):
    m = np.zeros((g.Y, g.X), dtype=bool)
    for y, x in points:
        m[max(0, y - reach):y + reach + 1, max(0, x - reach):x + reach + 1] = True
    return m


@pytest.mark.parametrize("name", list(SHAPES))
@pytest.mark.parametrize("prec", ["fp32", "bf16"])
def test_a_huge_mask_is_one_more_term(name, prec):
    """A pixel of 1e30, larger than any transform's rounding could hold: the
    outputs around it are its terms, the others those without it."""
    g, s, K = problem(**SHAPES[name])
    if prec == "bf16":  # exact in BF16, so that the oracle has the same products
        K = torch.tensor(K).bfloat16().double().numpy()
    r = g.k // 2
    rng = np.random.default_rng(1)
    c, y = (torch.tensor(rng.standard_normal(shape)).bfloat16().double().numpy()
            for shape in (g.c_shape(), g.y_shape()))
    py, px = g.Y // 2, g.X - 2
    cm, ym = c.copy(), y.copy()
    cm[:, py, px, 1], ym[:, py, px, 2:5] = 1e30, -1e30
    tol = (1e-2, 2e-2) if prec == "bf16" else (TOL, 1e-5)
    op = sw.Operator(g, K, s, precision=prec)
    try:
        clean = host(op.forward(dev(c))), host(op.adjoint(dev(y)))
        got = host(op.forward(dev(cm))), host(op.adjoint(dev(ym)))
        want = oracle.forward(g, s, K, cm), oracle.adjoint(g, s, K, ym)
        m = near(g, [(py, px)], r)
        for a, b, w in zip(got, clean, want):
            assert np.isfinite(a).all()
            assert rel(a[:, ~m], b[:, ~m]) <= TOL
            assert rel(a[:, m], w[:, m]) <= tol[0] + tol[1]
    finally:
        op.close()


@pytest.mark.parametrize("value", [np.inf, -np.inf, np.nan])
@pytest.mark.parametrize("name", list(SHAPES))
def test_a_call_leaves_no_marks_for_the_next(name, value):
    g, s, K = problem(**SHAPES[name])
    rng = np.random.default_rng(2)
    c, y = rng.standard_normal(g.c_shape()), rng.standard_normal(g.y_shape())
    op = sw.Operator(g, K, s)
    try:
        want = op.forward(dev(c)), op.adjoint(dev(y))
        cm, ym = c.copy(), y.copy()
        cm[0, 0, 0, 0] = ym[0, 0, 0, 0] = value
        for _ in range(3):
            op.forward(dev(cm))
            op.adjoint(dev(ym))
            assert torch.equal(op.forward(dev(c)), want[0])
            assert torch.equal(op.adjoint(dev(y)), want[1])
        # every output of an input without a finite value
        assert not torch.isfinite(op.forward(torch.full_like(dev(c), value))).any()
        assert not torch.isfinite(op.adjoint(torch.full_like(dev(y), value))).any()
    finally:
        op.close()


@pytest.mark.parametrize("value", [np.inf, np.nan, 3e38])
@pytest.mark.parametrize("kw", [dict(), dict(refine_every=2, refine_precision="fp32"),
                                dict(refine_every=2, refine_precision="fp32", refine_budget=0.05)])
@pytest.mark.parametrize("name", list(SHAPES))
def test_a_bad_pixel_keeps_its_neighbourhood(name, kw, value):
    """Three iterations of a solve (plain, refined on the host's and on the
    device's schedule): each gradient reaches 2 r further."""
    g, s, K = problem(**SHAPES[name])
    rng = np.random.default_rng(3)
    y = rng.standard_normal(g.y_shape())
    ym = y.copy()
    py, px, n = g.Y // 2, g.X // 2, 3
    ym[:, py, px, :] = value
    prm = sw.SolveParams(step=1e-4, lambda_l1=1e-3, lambda_tv=0.0, **kw)
    op = sw.Operator(g, K, s)
    try:
        out = []
        for data in (y, ym):
            op.fista_init(dev(data), prm)
            op.fista_step(n)
            out.append(host(op.fista_get()))
        m = near(g, [(py, px)], g.k // 2 * (1 + 2 * (n - 1)))
        assert not m.all()
        assert np.isfinite(out[1][:, ~m]).all()
        assert rel(out[1][:, ~m], out[0][:, ~m]) <= 1e-5
        # parameter gradient: NaN or infinite where a sum contains it
        if not np.isfinite(value):
            dk, dmu = op.param_grad(dev(np.abs(out[0])), dev(ym))
            assert not np.isfinite(dk).any()
    finally:
        op.close()


def test_an_infinity_in_the_iterate_stays_near_in_refined_increments():
    """H^T H of an increment that is infinite at one pixel, the measurements
    being finite: from a saved state whose c and momentum iterate hold it."""
    g, s, K = problem(**SHAPES["one_tile"])
    y = dev(np.random.default_rng(4).standard_normal(g.y_shape()))
    prm = sw.SolveParams(step=1e-4, lambda_l1=1e-3, lambda_tv=0.0, refine_every=100,
                         refine_precision="fp32")
    op = sw.Operator(g, K, s)
    try:
        op.fista_init(y, prm)
        op.fista_step(2)
        state = bytearray(op.fista_save())
        n = int(np.prod(g.c_shape()))
        sizes = np.frombuffer(state, dtype=np.uint8).size
        head = sizes - 4 * n * 4 - 16 * 8 - 4 * 4
        z = np.frombuffer(state, dtype=np.float32, count=n, offset=head + 2 * n * 4)
        op.fista_step(2)
        want = host(op.fista_get())
        py, px = g.Y // 2, g.X // 2
        zin = np.array(z).reshape(g.c_shape())
        zin[:, py, px, :] = np.inf  # the prox input: c, and so the increment, become infinite
        state[head + 2 * n * 4:head + 3 * n * 4] = zin.tobytes()
        op.fista_restore(bytes(state))
        op.fista_step(2)
        got = host(op.fista_get())
        m = near(g, [(py, px)], g.k // 2 * 2)
        assert np.isfinite(got[:, ~m]).all()
        assert rel(got[:, ~m], want[:, ~m]) <= 1e-5
        assert not np.isfinite(got[:, py, px]).all() or (got[:, py, px] == 0).any()
    finally:
        op.close()


@pytest.mark.parametrize("share", ["pixel", "all"])
def test_cost_of_bad_measurements(share):
    """A solve whose measurements hold NaNs at one pixel, or everywhere, takes
    no more than a few times a clean one (a direct sum per output of the image
    took thousands of times as long)."""
    g, s, K = problem(X=64, Y=60, Z=48, T=160, N=12, P=2, k=15, cycle=6)
    y = dev(np.random.default_rng(5).standard_normal(g.y_shape()))
    bad = y.clone()
    if share == "pixel":
        bad[:, 30, 30] = float("nan")
    else:
        bad[:] = float("nan")
    prm = sw.SolveParams(step=1e-6, lambda_l1=1e-3, lambda_tv=1e-3, inner_iters=5)
    op = sw.Operator(g, K, s)
    try:
        ms = []
        for data in (y, bad):
            op.fista_init(data, prm)
            op.fista_step(3)
            a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            a.record()
            op.fista_step(10)
            b.record()
            b.synchronize()
            ms.append(a.elapsed_time(b))
        print(share, ms)
        assert ms[1] <= 10 * ms[0]
    finally:
        op.close()
