"""The work that users of swopt have it do, as cases to be timed and compared.

Every case is one call, or one chain of calls, of the public Python binding:
the operators H and H^T at the precisions they are used at, H with its
gradients in c, kappa and mu, the proximal maps, whole solves, and a batch of
uneven problems.  Geometries are those of the repository's workloads (16 x 16
x 24 up to 128 x 128 x 96) and of its uneven batch problems, with odd sizes
among them.

Inputs are synthetic and come from the seed alone: a focused transducer's
per-depth kernel (aperture points on a spherical cap, spherical spreading, a
Gaussian-derivative impulse response), vessel-like tubes as concentrations,
and measurements H c plus noise at 20 dB, H taken here in 64 bits by FFTs.
"""
import functools
import math
from types import SimpleNamespace

import numpy as np
import torch

import paper_2510_23739_gb300 as sw

DX, DZ, DT, SOUND, FOCUS, APERTURE = 0.020, 0.010, 0.008, 1.5, 3.0, 1.5
KAPPA = {2: (0.05, 0.0), 3: (0.03, 0.08, 0.0)}
SNR_DB = 20.0


def _geom(X, Y, Z, T, N, cycle, P, k):
    return {"X": X, "Y": Y, "Z": Z, "T": T, "N": N, "cycle": cycle, "P": P, "k": k}


TINY = _geom(16, 16, 24, 64, 8, 8, 2, 7)
MEDIUM = _geom(64, 64, 64, 256, 40, 10, 2, 15)
LARGE = _geom(128, 128, 96, 512, 60, 10, 3, 31)
RAGGED = _geom(45, 37, 77, 209, 30, 10, 3, 13)


def listed():
    return [
        # the smallest call: one H c on the tiny workload, where launches and latency count
        {"name": "forward_tiny_fp32", "kind": "forward", "precision": "fp32", **TINY},
        # simulating data at the default precision (the accuracy reference), largest workload
        {"name": "forward_large_fp32", "kind": "forward", "precision": "fp32", **LARGE},
        # back-projection on a scan with no size that is a multiple of anything
        {"name": "adjoint_ragged_fp32", "kind": "adjoint", "precision": "fp32", **RAGGED},
        # simulating data on the largest grid in the solver's fast precision
        {"name": "forward_large_bf16", "kind": "forward", "precision": "bf16",
         **{**LARGE, "k": 15}},
        # back-projection of measurements on the medium workload, the same precision
        {"name": "adjoint_medium_bf16", "kind": "adjoint", "precision": "bf16", **MEDIUM},
        # learning kappa and mu: H and its backward through autograd, an uneven problem
        {"name": "gradient_uneven_bf16x3", "kind": "gradient", "precision": "bf16x3",
         **_geom(48, 48, 117, 336, 20, 10, 2, 15)},
        # the TV prox by itself (denoising): a volume that fits the SMs, and the largest
        {"name": "prox_tv_medium", "kind": "prox_tv", "precision": "fp32", "inner": 10, **MEDIUM},
        {"name": "prox_tv_large", "kind": "prox_tv", "precision": "fp32", "inner": 10,
         **{**LARGE, "k": 3, "T": 256}},
        # the prox of the full regulariser with the pulse-image term
        {"name": "prox_joint_uneven", "kind": "prox_joint", "precision": "fp32", "inner": 10,
         **_geom(96, 80, 77, 256, 40, 10, 3, 3)},
        # a short solve as a user starts one: default precision, medium workload
        {"name": "solve_medium_fp32", "kind": "solve", "precision": "fp32", "iters": 10,
         "inner": 10, **MEDIUM},
        # the refined BF16 solve on the largest grid, set up and stepped as a long run is
        {"name": "steps_large_refined", "kind": "steps", "precision": "bf16", "iters": 40,
         "inner": 10, **{**LARGE, "k": 15}},
        # several uneven problems stepped together
        {"name": "batch_refined", "kind": "batch", "precision": "bf16", "iters": 10, "inner": 10,
         "problems": 3, **_geom(32, 48, 64, 224, 30, 10, 2, 11)},
    ]


def draw(rng):
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["forward", "forward", "adjoint", "adjoint", "gradient", "prox_tv",
                       "prox_joint", "solve", "steps"])
    P = rng.choice([2, 3])
    cycle = rng.choice([4, 8, 10])
    Z = log_int(20, 120)
    precision = {"gradient": rng.choice(["fp32", "bf16x3"]), "solve": "fp32", "steps": "bf16",
                 "prox_tv": "fp32", "prox_joint": "fp32"}.get(
                     kind, rng.choice(["fp32", "fp32", "bf16", "bf16x3"]))
    # the widest supports at the accuracy reference's precision
    k = rng.choice([5, 7, 9, 11, 13, 15] + ([19, 23, 31] if precision == "fp32" else []))
    g = _geom(log_int(14, 120), log_int(14, 120), Z, log_int(max(64, 2 * Z), 480),
              cycle * rng.randint(1, 5), cycle, P, k)
    case = {"kind": kind, "precision": precision, **g}
    if kind in ("prox_tv", "prox_joint"):
        case.update(inner=rng.randint(4, 12), k=3)
    elif kind in ("solve", "steps"):
        # a fifth of the largest listed solve's work at most
        case.update(inner=rng.randint(4, 12), iters=rng.randint(3, 8))
        case.update({f: min(case[f], m) for f, m in (("X", 64), ("Y", 64), ("k", 15))})
    return case


# -- inputs -------------------------------------------------------------------

def _key(case):
    return tuple(case[f] for f in ("X", "Y", "Z", "T", "N", "cycle", "P", "k"))


def _geometry(key):
    X, Y, Z, T, N, cycle, P, k = key
    return SimpleNamespace(X=X, Y=Y, Z=Z, T=T, N=N, P=P, k=k, pulses_per_cycle=cycle, dz_mm=DZ)


def _switching(P):
    return SimpleNamespace(kappa=KAPPA[P], eps_bar=(1.0,) * (P - 1) + (0.0,),
                           eps_off=(0.0,) * (P - 1) + (1.0,), mu_per_mm=2.0)


@functools.lru_cache(maxsize=16)
def _kernel(Z, k, T):
    """K[Z][k][k][T] in 64 bits: 256 aperture points, arrivals binned, impulse response."""
    rng = np.random.default_rng(0)
    cos_max = math.cos(math.asin(APERTURE / FOCUS))
    ct = 1.0 - rng.random(256) * (1.0 - cos_max)
    phi = 2.0 * math.pi * rng.random(256)
    st = np.sqrt(np.maximum(0.0, 1.0 - ct * ct))
    px, py, pz = FOCUS * st * np.cos(phi), FOCUS * st * np.sin(phi), FOCUS * (1.0 - ct)
    cdt, r = SOUND * DT, k // 2
    gate = int(np.rint(FOCUS / cdt)) - T // 2
    off = np.arange(-r, r + 1) * DX
    lat = ((px - off[:, None]) ** 2)[None] + ((py - off[:, None]) ** 2)[:, None]  # [dy][dx][256]
    rows = np.arange(k * k)[:, None] * T
    q = np.zeros((Z, k * k * T))
    for j in range(Z):
        d = np.sqrt(lat + (pz - (FOCUS + (j - (Z - 1) / 2.0) * DZ)) ** 2).reshape(k * k, 256)
        t = np.rint(d / cdt).astype(np.int64) - gate
        ok = (t >= 0) & (t < T)
        q[j] = np.bincount((rows + t)[ok], weights=(1.0 / (4.0 * math.pi * 256 * d))[ok],
                           minlength=k * k * T)
    sigma = 1.0 / (2.0 * math.pi * 50.0)
    J = int(math.ceil(4.0 * sigma / DT))
    tau = np.arange(-J, J + 1) * DT
    v = -(tau / sigma ** 2) * np.exp(-tau ** 2 / (2.0 * sigma ** 2))
    v /= np.abs(v).max()
    q = q.reshape(Z, k, k, T)
    hit = np.nonzero(q.any(axis=(0, 1, 2)))[0]
    lo, hi = max(0, hit[0] - J), min(T, hit[-1] + J + 1)
    src = q[..., lo:hi].copy()
    K = np.zeros((Z, k, k, T))
    for s in range(-J, J + 1):
        a, b = max(lo, lo + s), min(hi, hi + s)
        K[..., a:b] += src[..., a - s - lo:b - s - lo] * v[s + J]
    return K


def _fft_len(n):
    while True:
        m = n
        for p in (2, 3, 5):
            while m % p == 0:
                m //= p
        if m == 1:
            return n
        n += 1


class _Model:
    """H and H^T in 64 bits by plain FFTs (torch), for making inputs and for exact()."""

    def __init__(self, key):
        self.key = key
        X, Y, Z, T, N, cycle, P, k = key
        r = k // 2
        K = _kernel(Z, k, T)
        hit = np.nonzero(K.any(axis=(0, 1, 2)))[0]
        self.lo, self.hi = int(hit[0]), int(hit[-1]) + 1
        self.L = (_fft_len(Y + r), _fft_len(X + r))
        tw = self.hi - self.lo
        self.Q = min(N, cycle)
        # u[y, x] = sum_d b[y + d] K[d]: a convolution with the kernel placed at -d
        Kd = torch.from_numpy(np.ascontiguousarray(K[..., self.lo:self.hi])).cuda()
        place = torch.zeros((Z, tw, *self.L), dtype=torch.float64, device="cuda")
        iy = (-(torch.arange(k, device="cuda") - r)) % self.L[0]
        ix = (-(torch.arange(k, device="cuda") - r)) % self.L[1]
        place[:, :, iy[:, None], ix[None, :]] = Kd.permute(0, 3, 1, 2)
        f = torch.fft.rfft2(place)
        self.Kf = f.permute(2, 3, 0, 1).reshape(-1, Z, tw).contiguous()  # [freq][j][t]

    def weights(self, kappa, mu):
        """S[m][p][j] of the Q states, differentiable in kappa and mu."""
        P, Z = self.key[6], self.key[2]
        s = _switching(P)
        eb = torch.tensor(s.eps_bar, dtype=torch.float64, device="cuda")[None, :, None]
        eo = torch.tensor(s.eps_off, dtype=torch.float64, device="cuda")[None, :, None]
        ph = torch.exp(-mu * torch.arange(Z, device="cuda", dtype=torch.float64) * DZ)
        m = torch.arange(self.Q, device="cuda", dtype=torch.float64)[:, None, None]
        return ph * (eb * torch.exp(-kappa[None, :, None] * ph * m) + eo)

    def default_weights(self):
        s = _switching(self.key[6])
        return self.weights(torch.tensor(s.kappa, dtype=torch.float64, device="cuda"),
                            torch.tensor(s.mu_per_mm, dtype=torch.float64, device="cuda"))

    def _spectrum(self, v):  # [Q][Y][X][C] -> [freq][Q][C]
        f = torch.fft.rfft2(v, s=self.L, dim=(1, 2))
        return f.permute(1, 2, 0, 3).reshape(-1, v.shape[0], v.shape[3])

    def _space(self, f):  # [freq][Q][C] -> [Q][Y][X][C]
        X, Y = self.key[0], self.key[1]
        f = f.reshape(self.L[0], self.L[1] // 2 + 1, f.shape[1], f.shape[2]).permute(2, 0, 1, 3)
        return torch.fft.irfft2(f, s=self.L, dim=(1, 2))[:, :Y, :X].contiguous()

    def acoustic(self, b):  # [Q][Y][X][Z] -> [Q][Y][X][window]
        return self._space(self._spectrum(b) @ self.Kf)

    def acoustic_t(self, u):  # [Q][Y][X][window] -> [Q][Y][X][Z]
        return self._space(self._spectrum(u) @ self.Kf.conj().transpose(1, 2))

    def forward_states(self, c):
        return self.acoustic(torch.einsum("mpj,pyxj->myxj", self.default_weights(), c.double()))

    def expand(self, u, dtype):  # states and window -> [N][Y][X][T]
        X, Y, Z, T, N, cycle, P, k = self.key
        y = torch.zeros((N, Y, X, T), dtype=dtype, device="cuda")
        for n in range(N):
            y[n, :, :, self.lo:self.hi] = u[n % cycle]
        return y

    def fold(self, y):  # [N][Y][X][T] -> pulses of one state summed, in the window
        N, cycle = self.key[4], self.key[5]
        return torch.stack([sum(y[n, :, :, self.lo:self.hi].double() for n in range(m, N, cycle))
                            for m in range(self.Q)])

    def adjoint(self, y):
        return torch.einsum("mpj,myxj->pyxj", self.default_weights(),
                            self.acoustic_t(self.fold(y)))

    @functools.cached_property
    def step(self):
        """1 / a bound of ||H||^2 (the largest singular value over the frequencies)."""
        v = torch.ones((self.Kf.shape[0], self.Kf.shape[2], 1), dtype=torch.complex128,
                       device="cuda")
        for _ in range(30):
            v = self.Kf.conj().transpose(1, 2) @ (self.Kf @ v)
            n = torch.linalg.vector_norm(v, dim=(1, 2), keepdim=True)
            v = v / n.clamp_min(1e-300)
        S, N, cycle = self.default_weights(), self.key[4], self.key[5]
        count = torch.tensor([len(range(m, N, cycle)) for m in range(self.Q)],
                             dtype=torch.float64, device="cuda")
        gram = torch.einsum("m,mpj,mqj->jpq", count, S, S)
        L = float(n.max()) * float(torch.linalg.matrix_norm(gram, ord=2).max())
        return float("%.3g" % (1.0 / L))


@functools.lru_cache(maxsize=2)
def _model(key):
    return _Model(key)


def _tubes(case, rng):
    """Vessel-like tubes: [P][Y][X][Z] on the GPU, values in [0, 1)."""
    X, Y, Z, T, N, cycle, P, k = _key(case)
    dev, c = "cuda", torch.zeros((P, Y, X, Z), dtype=torch.float32, device="cuda")
    pos = torch.stack(torch.meshgrid(torch.arange(Y, device=dev) * DX, torch.arange(X, device=dev) * DX,
                                     torch.arange(Z, device=dev) * DZ, indexing="ij"), dim=-1)
    ext = np.array([(Y - 1) * DX, (X - 1) * DX, (Z - 1) * DZ])
    for i in range(max(4, min(X, Y) // 2)):
        a, b = rng.random(3) * ext, rng.random(3) * ext
        radius, value, p = rng.uniform(1.0, 3.0) * DX, rng.uniform(0.5, 1.0), int(rng.integers(0, P))
        at = torch.tensor(a, dtype=torch.float32, device=dev)
        ab = torch.tensor(b - a, dtype=torch.float32, device=dev)
        t = ((pos - at) @ ab / float(max((b - a) @ (b - a), 1e-12))).clamp(0, 1)
        inside = (pos - at - t[..., None] * ab).norm(dim=-1) <= radius
        c[p] = torch.where(inside, c[p].clamp_min(value), c[p])
    return c


def _measurements(case, c, rng):
    """H c plus white noise at 20 dB, float32 [N][Y][X][T]."""
    M = _model(_key(case))
    y = M.expand(M.forward_states(c), torch.float32)
    power = float(y.double().square().mean())
    gen = torch.Generator(device="cuda").manual_seed(int(rng.integers(1 << 31)))
    noise = torch.empty_like(y).normal_(generator=gen)
    return y.add_(noise, alpha=math.sqrt(power / 10 ** (SNR_DB / 10)))


def _inputs(case, seed):
    """What the seed decides: (c, y or None, ...) as the case's kind needs them."""
    rng = np.random.default_rng(seed)
    c = _tubes(case, rng)
    kind = case["kind"]
    if kind in ("prox_tv", "prox_joint"):
        # a gradient step's output: tubes in noise
        gen = torch.Generator(device="cuda").manual_seed(int(rng.integers(1 << 31)))
        return c + 0.2 * torch.empty_like(c).normal_(generator=gen), None
    y = _measurements(case, c, rng) if kind in ("adjoint", "gradient", "solve", "steps") else None
    return c, y


def _params(case):
    refined = sw.REFINED_DEFAULTS if case["precision"] != "fp32" else {}
    return sw.SolveParams(step=_model(_key(case)).step, lambda_l1=1e-3, lambda_tv=1e-3,
                          inner_iters=case["inner"], max_iters=case["iters"], **refined)


def _operator(case):
    key = _key(case)
    return sw.Operator(_geometry(key), _kernel(key[2], key[7], key[3]), _switching(key[6]),
                       precision=case["precision"])


def _problems(case):
    """The uneven problems of a batch case, of growing size."""
    out = []
    for i in range(case["problems"]):
        out.append({**case, "kind": "steps", "X": case["X"] + 17 * i, "Y": case["Y"] - 7 * i,
                    "Z": case["Z"] + 11 * i, "T": case["T"] + 24 * i, "k": case["k"] + 2 * i})
    return out


def prepare(case, seed):
    kind = case["kind"]
    s = SimpleNamespace(case=case, kind=kind)
    if kind == "batch":
        s.parts = [prepare(q, 100 * seed + i) for i, q in enumerate(_problems(case))]
        return s
    s.c, s.y = _inputs(case, seed)
    if kind in ("solve", "steps"):
        s.params, s.c = _params(case), None
    s.op = _operator(case)
    if kind == "gradient":
        w = _switching(case["P"])
        s.c.requires_grad_()
        s.kappa = torch.tensor(w.kappa, dtype=torch.float32, requires_grad=True)
        s.mu = torch.tensor(w.mu_per_mm, dtype=torch.float32, requires_grad=True)
    elif kind == "prox_joint":
        s.step2 = 1.0 / s.op.prox_joint_step_bound(*_JOINT)
    return s


_JOINT = (0.3, 0.1, 0.2)  # lambda_tv, lambda_l1, lambda_3 of the joint prox


def run(s):
    kind = s.kind
    if kind == "forward":
        return s.op.forward(s.c)
    if kind == "adjoint":
        return s.op.adjoint(s.y)
    if kind == "gradient":
        y = sw.HFunction.apply(s.c, s.kappa, s.mu, s.op)
        # the measurements are pulled back: a residual y - data would hand y's
        # rounding to everything that follows
        return y.detach(), torch.autograd.grad(y, (s.c, s.kappa, s.mu), grad_outputs=s.y)
    if kind == "prox_tv":
        return s.op.prox_tv(s.c, 0.1, s.case["inner"])
    if kind == "prox_joint":
        return s.op.prox_joint(s.c, 0.5, *_JOINT, s.case["inner"], s.step2)
    if kind == "solve":
        c, stats = s.op.solve(s.y, s.params)
        return c, stats["objective"], stats["data_fit"]
    if kind == "steps":
        s.op.fista_init(s.y, s.params)
        s.op.fista_step(s.case["iters"])
        return s.op.fista_get()
    for p in s.parts:
        p.op.fista_init(p.y, p.params)
    batch = sw.Batch([p.op for p in s.parts])
    batch.step(s.case["iters"])
    out = [p.op.fista_get() for p in s.parts]
    batch.close()
    return out


def work(case):
    """Inputs read once and outputs written once; the operations of the method as the
    sums define it: two per nonzero kernel entry, state and position for H or H^T."""
    if case["kind"] == "batch":
        parts = [work(q) for q in _problems(case)]
        return {f: sum(p[f] for p in parts) for f in ("bytes", "flops")}
    X, Y, Z, T, N, cycle, P, k = _key(case)
    nc, ny = 4.0 * P * Y * X * Z, 4.0 * N * Y * X * T
    kind = case["kind"]
    if kind == "prox_tv":
        return {"bytes": 2 * nc, "flops": 20.0 * case["inner"] * P * Y * X * Z}
    if kind == "prox_joint":
        return {"bytes": 2 * nc, "flops": 20.0 * case["inner"] * (P + min(N, cycle)) * Y * X * Z}
    H = 2.0 * min(N, cycle) * X * Y * np.count_nonzero(_kernel(Z, k, T))
    if kind in ("forward", "adjoint"):
        return {"bytes": nc + ny, "flops": H}
    if kind == "gradient":
        return {"bytes": 2 * (nc + ny), "flops": 2 * H}
    # one H and one H^T per iteration and for the first gradient; the measurements once
    return {"bytes": nc + ny, "flops": 2 * H * (case["iters"] + 1)}


# -- what run() returns, in 64 bits --------------------------------------------

def _div_t(q):
    """D^T q for q [3][P][Y][X][Z], D the forward differences along y, x, z."""
    out = torch.zeros_like(q[0])
    for a, dim in enumerate((1, 2, 3)):
        n = out.shape[dim] - 1
        if n < 1:
            continue
        e = q[a].narrow(dim, 0, n)
        out.narrow(dim, 1, n).add_(e)
        out.narrow(dim, 0, n).sub_(e)
    return out


def _diff(x):
    out = torch.zeros((3, *x.shape), dtype=x.dtype, device=x.device)
    for a, dim in enumerate((1, 2, 3)):
        n = x.shape[dim] - 1
        if n >= 1:
            out[a].narrow(dim, 0, n).copy_(x.narrow(dim, 1, n) - x.narrow(dim, 0, n))
    return out


def _betas(n):
    t = 1.0
    for _ in range(n):
        t1 = 0.5 * (1.0 + math.sqrt(1.0 + 4.0 * t * t))
        yield (t - 1.0) / t1
        t = t1


def _prox_tv(z, tau, inner):
    r = torch.zeros((3, *z.shape), dtype=torch.float64, device="cuda")
    u = torch.zeros_like(r)
    for beta in _betas(inner):
        un = (r + _diff(z - _div_t(r)) / 12.0).clamp(-tau, tau)
        r = un + beta * (un - u)
        u = un
    return z - _div_t(u)


def _prox_joint(M, z, alpha, lams, inner, step2):
    """Algorithm 2 on the dual of the full regulariser with c >= 0, one dual per state."""
    tv, l1, l3 = lams
    X, Y, Z, T, N, cycle, P, k = M.key
    S = M.default_weights()
    C = torch.tensor([len(range(m, N, cycle)) for m in range(M.Q)], dtype=torch.float64,
                     device="cuda")

    def lift(w):
        return [tv * _diff(w), l1 * w, l3 * _diff(torch.einsum("mpj,pyxj->myxj", S, w))]

    def lower(d):
        b = _div_t(d[2]) * C[:, None, None, None]
        return tv * _div_t(d[0]) + l1 * d[1] + l3 * torch.einsum("mpj,myxj->pyxj", S, b)

    shape = [(3, P, Y, X, Z), (P, Y, X, Z), (3, M.Q, Y, X, Z)]
    r = [torch.zeros(s, dtype=torch.float64, device="cuda") for s in shape]
    u = [torch.zeros_like(v) for v in r]
    for beta in _betas(inner):
        w = (z - lower(r)).clamp_min(0)
        un = [(a + step2 * b).clamp(-alpha, alpha) for a, b in zip(r, lift(w))]
        r = [a + beta * (a - b) for a, b in zip(un, u)]
        u = un
    return (z - lower(u)).clamp_min(0)


def exact(case, seed):
    kind = case["kind"]
    if kind in ("solve", "steps", "batch"):
        return None
    c, y = _inputs(case, seed)
    if kind == "prox_tv":
        return _prox_tv(c.double(), 0.1, case["inner"])
    M = _model(_key(case))
    if kind == "prox_joint":
        S, N, cycle = M.default_weights(), case["N"], case["cycle"]
        C = torch.tensor([len(range(m, N, cycle)) for m in range(M.Q)], dtype=torch.float64,
                         device="cuda")
        peak = (S.square().sum(1).max(1).values * C).sum()
        tv, l1, l3 = _JOINT
        step2 = 1.0 / float(12 * tv * tv + l1 * l1 + 12 * l3 * l3 * peak)
        return _prox_joint(M, c.double(), 0.5, _JOINT, case["inner"], step2)
    if kind == "forward":
        return M.expand(M.forward_states(c), torch.float64)
    if kind == "adjoint":
        return M.adjoint(y)
    w = _switching(case["P"])
    kappa = torch.tensor(np.float32(w.kappa).astype(np.float64), device="cuda", requires_grad=True)
    mu = torch.tensor(float(np.float32(w.mu_per_mm)), dtype=torch.float64, device="cuda",
                      requires_grad=True)
    S = M.weights(kappa, mu)
    g = M.acoustic_t(M.fold(y))  # A^T of the cotangent, per state
    with torch.no_grad():
        u = M.acoustic(torch.einsum("mpj,pyxj->myxj", S, c.double()))
        gc = torch.einsum("mpj,myxj->pyxj", S, g)
    W = torch.einsum("myxj,pyxj->mpj", g, c.double())
    gk, gm = torch.autograd.grad((W * S).sum(), (kappa, mu))
    return M.expand(u, torch.float64), (gc, gk, gm)
