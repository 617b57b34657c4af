"""Measured cases of the many-chain surrogate mMALA sampler, through its public calls.

A case is one thing that a user of the library has it do over and over: advance
a pool of chains and read it, run a short ensemble from host fields, evaluate a
surrogate and its Jacobian in place, or assess recorded chains.  `listed()`
gives the fixed ones, `draw()` others of the same ranges; `prepare()` makes the
inputs and the handles, `run()` is one pass, `work()` what a pass cannot do
without and `exact()` the same results in float64 from plain torch.

Results of the tensor-core precision are kept as float32, the precision that
path delivers; what it holds in float64 (positions encoded from a field) and
every result of the float64 path stay float64.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2403_08220_gb300 as dino

GAMMA, DELTA = 0.1, 1.0          # prior (delta I - gamma Laplacian)^-2
ACTS = {"identity": 0, "tanh": 1, "gelu": 2}
MAPS = {"auto": 0, "cholesky": 1, "perturbation": 2, "eigen": 3}
MAX_PERTURBATION_DY = 192        # above it (or with d_y >= r) "auto" is the Cholesky map


def _step(name, precision, basis, n_grid, widths, act, chains, steps, **more):
    c = dict(name=name, kind="step", precision=precision, basis=basis, n_grid=n_grid,
             widths=widths, act=act, noise_map="auto", chains=chains, steps=steps, dt=0.5,
             noise_frac=0.01, start="prior")
    c.update(more)
    return c


def listed():
    r200 = "200-400-400-100"
    return [
        # a small posterior explored by few chains in the plain float64 path at a step
        # size that mixes: the smallest calls, one after the other
        _step("fp64_small_c64", "fp64", "kle", 33, "16-64-64-49", "tanh", 64, 50, dt=0.002,
              noise_map="cholesky"),
        # the float64 path of the r = 200 posterior: reference runs, and data too precise
        # for the tensor path
        _step("fp64_r200_c1024", "fp64", "kle", 65, r200, "gelu", 1024, 2),
        # the r = 200 posterior on the tensor path with a pool of the size one analyst runs
        _step("bf16_r200_c64", "bf16", "explicit", 65, r200, "gelu", 64, 10),
        # the same with the large ensemble: the throughput the library is built for
        _step("bf16_r200_c16384", "bf16", "explicit", 65, r200, "gelu", 16384, 10),
        # a mixing chain (data less informative, start near the truth): accepted proposals
        # update the field, which is read back
        _step("bf16_r200_mixing_c256", "bf16", "explicit", 65, r200, "gelu", 256, 8, dt=0.01,
              noise_frac=0.3, start="truth", field=True),
        # the paper's network: six hidden layers of 400, 25 observations, 41 x 41 field
        _step("bf16_paper_c4096", "bf16", "explicit", 41, "200" + "-400" * 6 + "-25", "gelu",
              4096, 10, start="truth"),
        # the paper's noise map (symmetric root from an eigendecomposition) on that network
        _step("bf16_eigen_c1024", "bf16", "explicit", 41, "200" + "-400" * 6 + "-25", "gelu",
              1024, 2, noise_map="eigen", start="truth"),
        # posteriors with at least as many observations as reduced dimensions
        # (two of the heterogeneous batch): a middling and its largest
        _step("bf16_r128_dy200_c4096", "bf16", "explicit", 65, "128-256-256-200", "gelu", 4096, 4),
        _step("bf16_r400_dy400_c512", "bf16", "explicit", 65, "400-800-800-400", "gelu", 512, 4),
        # a short ensemble run whole: host fields in, a few transitions, positions and
        # fields back, the pool freed
        _step("bf16_ensemble_c2048", "bf16", "explicit", 65, r200, "gelu", 2048, 4,
              kind="ensemble", start="truth", field=True),
        # the surrogate and its Jacobian at a few points on the caller's own device buffers
        dict(name="jacobian_noalloc_n8", kind="noalloc", widths=r200, act="gelu", points=8),
        # assessing ten recorded chains: effective sample sizes and the MPSRF
        dict(name="diagnostics_d200", kind="diag", dofs=200, chains=10, samples=1000, rho=0.9),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["wb", "wb", "wb", "square", "square", "fp64", "fp64", "eigen", "ensemble",
                       "noalloc", "diag"])
    if kind == "diag":
        dofs = rng.randint(8, 200)
        return dict(kind="diag", dofs=dofs, chains=rng.randint(2, 16),
                    samples=_log_int(rng, 50, 1000), rho=round(rng.uniform(0.3, 0.95), 3))
    if kind == "noalloc":
        r, dy = rng.randint(8, 256), rng.randint(4, 128)
        hidden = [rng.randint(16, 400) for _ in range(rng.randint(1, 4))]
        points = rng.randint(1, max(1, min(8, (1 << 20) // (2 * dy * max(hidden)))))
        return dict(kind="noalloc", widths="-".join(map(str, [r] + hidden + [dy])),
                    act=rng.choice(["tanh", "gelu"]), points=points)
    n_grid = rng.randint(17, 65)
    cap = min(n_grid * n_grid, 400)
    noise_map, precision = "auto", "bf16"
    if kind in ("wb", "ensemble"):
        r = rng.randint(24, min(cap, 256))
        dy = rng.randint(16, min(r - 1, 128))
    elif kind == "eigen":
        r = rng.randint(24, min(cap, 256))
        dy = rng.randint(16, min(r - 1, 40))
        noise_map = "eigen"
    elif kind == "square":
        r = _log_int(rng, 48, cap)
        dy = rng.randint(r, 400)
    else:
        precision = "fp64"
        r = _log_int(rng, 12, min(cap, 208))
        dy = rng.randint(4, 128)
    q = max(r, dy)      # hidden layers at least as wide as the reduced input and the output
    hidden = [rng.randint(q, 2 * q) for _ in range(rng.randint(1, 6))]
    w = [r] + hidden + [dy]
    # chains spread over the logarithm, within the work that the largest listed cases take
    per = min(r, dy) * sum(a * b for a, b in zip(w[1:-1], w[2:])) + dy * w[0] * w[1] + r * dy * dy
    limit = {"wb": 4e12, "ensemble": 4e11, "square": 2.5e11, "fp64": 4e10, "eigen": 2e11}[kind]
    most = {"wb": 16384, "ensemble": 2048, "square": 4096, "fp64": 1024, "eigen": 1024}[kind]
    steps = rng.randint(1, 4) if kind in ("eigen", "fp64", "square") else rng.randint(2, 10)
    most = max(16, min(most, int(limit / (per * steps))))
    c = _step("", precision, "kle" if precision == "fp64" else "explicit", n_grid,
              "-".join(map(str, w)), rng.choice(["gelu", "gelu", "tanh"]),
              _log_int(rng, 16, most), steps, noise_map=noise_map)
    del c["name"]
    if kind in ("wb", "eigen", "ensemble"):
        c.update(start="truth")
    if kind == "ensemble":
        c.update(kind="ensemble", field=True)
    return c


# ---- inputs ---------------------------------------------------------------------


def _widths(case):
    return [int(x) for x in case["widths"].split("-")]


def _gen(seed, device="cuda"):
    return torch.Generator(device=device).manual_seed(int(seed))


def _randn(g, *shape):
    return torch.randn(*shape, generator=g, device=g.device, dtype=torch.float64)


def _weights(widths, g):
    """LeCun-normal weights and N(0, 0.1^2) biases."""
    Ws = [_randn(g, o, i) / math.sqrt(i) for i, o in zip(widths[:-1], widths[1:])]
    return Ws, [0.1 * _randn(g, o) for o in widths[1:]]


def _act(kind, z):
    """Activation and its derivative."""
    if kind == "tanh":
        t = torch.tanh(z)
        return t, 1.0 - t * t
    if kind == "gelu":
        cdf = 0.5 * (1.0 + torch.erf(z * math.sqrt(0.5)))
        return z * cdf, cdf + z * torch.exp(-0.5 * z * z) / math.sqrt(2.0 * math.pi)
    return z, torch.ones_like(z)


def _forward(Ws, bs, act, x):
    ds = []
    for W, b in zip(Ws[:-1], bs[:-1]):
        x, d = _act(act, x @ W.T + b)
        ds.append(d)
    return x @ Ws[-1].T + bs[-1], ds


def _spectrum(n):
    """Sine matrix S and sqrt(lambda) on the n x n grid of modes [ky, kx]."""
    k = torch.arange(1, n + 1, dtype=torch.float64, device="cuda")
    h = 1.0 / (n + 1)
    S = math.sqrt(2.0 * h) * torch.sin(torch.outer(k, k) * (math.pi * h))
    kap = 4.0 / h ** 2 * torch.sin(0.5 * math.pi * h * k) ** 2
    return S, 1.0 / (DELTA + GAMMA * (kap[:, None] + kap[None, :]))


def _spectral(S, diag, X):
    """S (diag * (S X S)) S for fields X (..., N), nodes i + n j."""
    n = S.shape[0]
    Y = S @ X.reshape(X.shape[:-1] + (n, n)) @ S
    return (S @ (diag * Y) @ S).reshape(X.shape)


def _basis(case, r, seed):
    """Encoder E (r x N) and decoder D (N x r) on the device."""
    n = case["n_grid"]
    S, sq = _spectrum(n)
    if case["basis"] == "kle":
        kap = (1.0 / sq).cpu().numpy()
        ky, kx = np.meshgrid(np.arange(n), np.arange(n), indexing="ij")
        order = np.lexsort((kx.ravel(), np.round(kap, 9).ravel()))[:r]
        idx = torch.from_numpy(order).cuda()
        vy, vx = S[idx // n], S[idx % n]
        eta = (vy[:, :, None] * vx[:, None, :]).reshape(r, n * n)
        lam = sq.reshape(-1)[idx]
        return eta / lam[:, None], (eta * lam[:, None]).T.contiguous()
    # a derivative-informed basis: C_pr^-1-orthonormal columns, as a trained one is
    Q = torch.linalg.qr(_randn(_gen(seed * 7 + 1), n * n, r))[0].T.contiguous()
    return _spectral(S, 1.0 / sq, Q), _spectral(S, sq, Q).T.contiguous()


class _Posterior:
    """Weights, basis, data and starting fields of a case, from its seed."""

    def __init__(self, case, seed):
        self.widths = _widths(case)
        r, dy = self.widths[0], self.widths[-1]
        g = _gen(seed * 7 + 2)
        self.Ws, self.bs = _weights(self.widths, g)
        self.act = case["act"]
        truth = _randn(g, r)
        f, _ = _forward(self.Ws, self.bs, self.act, truth[None])
        sigma = case["noise_frac"] * float(torch.sqrt(torch.mean(f * f)))
        self.y = f[0] + sigma * _randn(g, dy)
        self.noise_var = sigma * sigma
        self.E, self.D = _basis(case, r, seed)
        self.S, self.sq = _spectrum(case["n_grid"])
        self.chain_seed = 1000003 + seed
        if case["start"] == "truth":
            # prior draws outside the reduced basis, near the truth inside it
            M = self.prior(_randn(g, case["chains"], case["n_grid"] ** 2))
            x = truth + 0.05 * _randn(g, case["chains"], r)
            self.m0 = M + (x - M @ self.E.T) @ self.D.T
        else:
            self.m0 = None

    def prior(self, z):
        n = self.S.shape[0]
        X = self.sq * z.reshape(-1, n, n)
        return (self.S @ X @ self.S).reshape(z.shape)


class _State:
    pass


def _np(t):
    return t.cpu().numpy()


def prepare(case, seed):
    s = _State()
    s.case = case
    if case["kind"] == "noalloc":
        s.widths = _widths(case)
        g = _gen(seed)
        s.Ws, s.bs = _weights(s.widths, g)
        s.x = _randn(g, case["points"], s.widths[0])
        s.f = torch.empty(case["points"], s.widths[-1], dtype=torch.float64, device="cuda")
        s.J = torch.empty(case["points"], s.widths[-1], s.widths[0], dtype=torch.float64,
                          device="cuda")
        return s
    s.ctx = dino.dino_init(torch.cuda.current_device())
    if case["kind"] == "diag":
        X = _np(_trajectory(case, seed))
        s.diag = dino.dino_diag_create(s.ctx, case["chains"], case["dofs"], case["samples"])
        for j in range(case["samples"]):
            dino.dino_diag_push(s.ctx, s.diag, X[j])
        return s
    p = _Posterior(case, seed)
    bf16 = case["precision"] == "bf16"
    explicit = case["basis"] == "explicit"
    s.r, s.N, s.seed = p.widths[0], case["n_grid"] ** 2, p.chain_seed
    s.sid = dino.dino_load_surrogate(
        s.ctx, n_grid=case["n_grid"], prior_gamma=GAMMA, prior_delta=DELTA, r=s.r,
        widths=p.widths, activation=ACTS[p.act], W=[_np(W) for W in p.Ws],
        b=[_np(b) for b in p.bs],
        basis_kind=dino.DINO_BASIS_EXPLICIT if explicit else dino.DINO_BASIS_KLE,
        E=_np(p.E) if explicit else None, D=_np(p.D) if explicit else None, y=_np(p.y),
        noise_var=p.noise_var, precision=dino.DINO_PREC_BF16 if bf16 else dino.DINO_PREC_FP64,
        noise_map=MAPS[case["noise_map"]])
    s.m0 = None if p.m0 is None else _np(p.m0)
    if case["kind"] == "step":
        s.pool = dino.dino_chains_create(s.ctx, s.sid, case["chains"], case["dt"], s.seed, m0=s.m0)
        s.m0 = None
    return s


# ---- one pass ---------------------------------------------------------------------


def _kept(case, out):
    """The pool's results as a user keeps them: float32 from the tensor path."""
    if case["precision"] == "fp64":
        return out
    wide = ("log_u", "m_r") if case["kind"] == "ensemble" else ("log_u",)
    return {k: torch.from_numpy(v).float() if v.dtype == np.float64 and k not in wide else v
            for k, v in out.items()}


def _read(case, s, pool):
    C = case["chains"]
    out = dino.dino_chains_read(s.ctx, pool, C, s.r, s.N, field=case.get("field", False))
    out.update(dino.dino_chains_read_last(s.ctx, pool, C, s.r))
    out["accepts"] = out["accepts"].astype(np.int64)
    return _kept(case, {k: v for k, v in out.items() if v is not None})


def run(s):
    case = s.case
    if case["kind"] == "noalloc":
        dino.dino_surrogate_jacobian_noalloc(
            case["points"], s.widths, ACTS[case["act"]], [W.data_ptr() for W in s.Ws],
            [b.data_ptr() for b in s.bs], s.x.data_ptr(), s.f.data_ptr(), s.J.data_ptr(),
            torch.cuda.current_stream().cuda_stream)
        return dict(f=s.f, J=s.J)
    if case["kind"] == "diag":
        out = dino.dino_diag_compute(s.ctx, s.diag, case["dofs"])
        return {k: np.asarray(out[k], dtype=np.float64)
                for k in ("ess", "ess_median", "msj", "mpsrf_w", "trace_w", "trace_v")}
    if case["kind"] == "ensemble":
        pool = dino.dino_chains_create(s.ctx, s.sid, case["chains"], case["dt"], s.seed, m0=s.m0)
        dino.dino_chains_step(s.ctx, pool, case["steps"], stats=False)
        out = _read(case, s, pool)
        dino.dino_chains_destroy(s.ctx, pool)
        return out
    dino.dino_chains_step(s.ctx, s.pool, case["steps"], stats=False)
    return _read(case, s, s.pool)


# ---- what a pass cannot do without --------------------------------------------------


def work(case):
    """Bytes: inputs, chain state and weights read once, results written once.  Flops: the
    network, its Jacobian in the cheaper order, the smaller Gram matrix and factor, the
    proposal's products, the prior draw and the two projections, per chain and transition."""
    if case["kind"] == "diag":
        d, k, n = case["dofs"], case["chains"], case["samples"]
        return dict(bytes=8.0 * (d * k * n + d), flops=2.0 * d * d * k * n / 2 + 20.0 * d ** 3)
    w = _widths(case)
    r, dy = w[0], w[-1]
    mlp = 2.0 * sum(a * b for a, b in zip(w[:-1], w[1:]))
    rev = 2.0 * dy * sum(a * b for a, b in zip(w[:-2], w[1:-1]))
    fwd = 2.0 * r * sum(a * b for a, b in zip(w[1:-1], w[2:]))
    weights = sum(a * b + b for a, b in zip(w[:-1], w[1:]))
    if case["kind"] == "noalloc":
        n = case["points"]
        return dict(bytes=8.0 * (weights + n * (r + dy + dy * r)), flops=n * (mlp + min(rev, fwd)))
    e = 8 if case["precision"] == "fp64" else 4
    n, N, C, T = case["n_grid"], case["n_grid"] ** 2, case["chains"], case["steps"]
    q = min(r, dy)
    flops = (mlp + min(rev, fwd) + r * dy * (q + 1) + q ** 3 / 3.0 + 6.0 * r * dy + 4.0 * q * q
             + 4.0 * n ** 3 + 4.0 * r * N)
    state = 2 * r * e + q * (q + 1) / 2 * 8 + (r * dy * e if dy < r else 0)
    nbytes = e * (weights + 2 * r * N) + C * (state + 8.0 * (3 * r + 4))
    if case.get("field"):
        nbytes += C * N * (e + 8.0)
    if case["kind"] == "ensemble":
        flops += 2.0 * r * N / T + (mlp + min(rev, fwd) + r * dy * (q + 1) + q ** 3 / 3.0) / T
        nbytes += C * N * 8.0
    return dict(bytes=nbytes, flops=C * T * flops)


# ---- the same results in float64 ------------------------------------------------------


def _philox(seed, stream, step, chains, blocks):
    """Philox4x32-10 words (chains, blocks, 4) as int64, counter (block, step, chain, stream)."""
    mask = 0xFFFFFFFF

    def mul(a, x):   # high and low words of the 64-bit product, by 16-bit pieces of a
        lo, hi = (a & 0xFFFF) * x, (a >> 16) * x
        mid = (lo >> 16) + hi
        return mid >> 16, ((mid & 0xFFFF) << 16) | (lo & 0xFFFF)

    c0 = torch.arange(blocks, device="cuda").expand(chains, blocks)
    c2 = torch.arange(chains, device="cuda")[:, None].expand(chains, blocks)
    c1, c3 = torch.full_like(c0, step), torch.full_like(c0, stream)
    k0, k1 = seed & mask, seed >> 32
    for _ in range(10):
        h0, l0 = mul(0xD2511F53, c0)
        h1, l1 = mul(0xCD9E8D57, c2)
        c0, c1, c2, c3 = h1 ^ c1 ^ k0, l1, h0 ^ c3 ^ k1, l0
        k0, k1 = (k0 + 0x9E3779B9) & mask, (k1 + 0xBB67AE85) & mask
    return torch.stack([c0, c1, c2, c3], -1)


def _normals(seed, stream, step, chains, count):
    u = (_philox(seed, stream, step, chains, (count + 3) // 4).double() + 0.5) * 2.0 ** -32
    r0, r1 = torch.sqrt(-2.0 * torch.log(u[..., 0])), torch.sqrt(-2.0 * torch.log(u[..., 2]))
    t0, t1 = 2.0 * math.pi * u[..., 1], 2.0 * math.pi * u[..., 3]
    z = torch.stack([r0 * torch.cos(t0), r0 * torch.sin(t0), r1 * torch.cos(t1),
                     r1 * torch.sin(t1)], -1)
    return z.reshape(chains, -1)[:, :count]


def _jacobian(Ws, ds):
    """df/dx (points, d_y, r) in reverse order from the activation derivatives."""
    P = Ws[-1].expand(ds[0].shape[0] if ds else 1, -1, -1)
    for W, d in zip(reversed(Ws[:-1]), reversed(ds)):
        P = (P * d[:, None, :]) @ W
    return P


def _mv(A, x):
    return (A @ x[..., None])[..., 0]


class _Geometry:
    """Misfit, K = J / sigma and the factor of the smaller of I + K K^T, I + K^T K."""

    def __init__(self, p, x):
        f, ds = _forward(p.Ws, p.bs, p.act, x)
        sigma = math.sqrt(p.noise_var)
        self.K = _jacobian(p.Ws, ds) / sigma
        self.eps = (f - p.y) / sigma
        self.phi = 0.5 * (self.eps ** 2).sum(-1)
        dy, r = self.K.shape[1:]
        self.small = dy < r
        G = self.K @ self.K.mT if self.small else self.K.mT @ self.K
        self.M = G + torch.eye(G.shape[-1], dtype=G.dtype, device=G.device)
        self.L = torch.linalg.cholesky(self.M)
        self.hld = torch.log(torch.diagonal(self.L, dim1=-2, dim2=-1)).sum(-1)

    def solve(self, x):
        """(I + H)^-1 x, H = K^T K."""
        if self.small:
            t = torch.cholesky_solve(_mv(self.K, x)[..., None], self.L)[..., 0]
            return x - _mv(self.K.mT, t)
        return torch.cholesky_solve(x[..., None], self.L)[..., 0]

    def log_rho0(self, m1, m2, dt, sc):
        """log of the surrogate mMALA proposal density over the pCN one, from m1 to m2."""
        q = _mv(self.K, m1) - self.eps
        w = _mv(self.K.mT, q)
        mhat = (m2 - sc * m1) / math.sqrt(1.0 - sc * sc)
        return (-dt / 8.0 * (w * self.solve(w)).sum(-1) + math.sqrt(dt) / 2.0 * (mhat * w).sum(-1)
                + self.hld - 0.5 * (_mv(self.K, mhat) ** 2).sum(-1))


def _noise(g, noise_map, xi, xi2):
    if noise_map == "eigen":
        lam, U = torch.linalg.eigh(g.M)
        root = torch.sqrt(lam)
        t = _mv(U, -_mv(U.mT, _mv(g.K, xi)) / (root * (1.0 + root)))
        return xi + _mv(g.K.mT, t)
    if noise_map == "perturbation":
        return g.solve(xi + _mv(g.K.mT, xi2))
    L = g.L
    if g.small:  # the Cholesky map factors I + K^T K
        r = xi.shape[-1]
        L = torch.linalg.cholesky(torch.eye(r, dtype=xi.dtype, device=xi.device) + g.K.mT @ g.K)
    return torch.linalg.solve_triangular(L.mT, xi[..., None], upper=True)[..., 0]


def _exact_chains(case, seed):
    p = _Posterior(case, seed)
    C, dt, N = case["chains"], case["dt"], case["n_grid"] ** 2
    r, dy = p.widths[0], p.widths[-1]
    sc = (4.0 - dt) / (4.0 + dt)
    cs = math.sqrt(1.0 - sc * sc)
    noise_map = case["noise_map"]
    if noise_map == "auto":
        noise_map = "perturbation" if dy < r and dy <= MAX_PERTURBATION_DY else "cholesky"
    m = p.m0 if p.m0 is not None else p.prior(_normals(p.chain_seed, 3, 0, C, N))
    a = m @ p.E.T
    ga = _Geometry(p, a)
    accepts = torch.zeros(C, dtype=torch.int64, device="cuda")
    for j in range(case["steps"]):
        xi = _normals(p.chain_seed, 0, j, C, r)
        xi2 = _normals(p.chain_seed, 4, j, C, dy) if noise_map == "perturbation" else None
        log_u = torch.log((_philox(p.chain_seed, 1, j, C, 1)[:, 0, 0].double() + 0.5) * 2.0 ** -32)
        mu = a - (1.0 - sc) * ga.solve(a + _mv(ga.K.mT, ga.eps))
        b = mu + cs * _noise(ga, noise_map, xi, xi2)
        gb = _Geometry(p, b)
        log_rho = ga.phi - gb.phi + gb.log_rho0(b, a, dt, sc) - ga.log_rho0(a, b, dt, sc)
        acc = log_u <= torch.clamp(log_rho, max=0.0)
        if bool(acc.any()):
            M = p.prior(_normals(p.chain_seed, 2, j, C, N))
            full = sc * m + cs * M
            full = full + (b - full @ p.E.T) @ p.D.T
            m, a = torch.where(acc[:, None], full, m), torch.where(acc[:, None], b, a)
            for k in ("K", "eps", "phi", "M", "L", "hld"):
                x, y = getattr(ga, k), getattr(gb, k)
                setattr(ga, k, torch.where(acc.reshape((C,) + (1,) * (x.dim() - 1)), y, x))
        accepts += acc
        del gb
    out = dict(m=m if case.get("field") else None, m_r=a, phi=ga.phi, accepts=accepts, b=b,
               mu=mu, log_rho=log_rho, log_u=log_u, accepted=acc)
    return {k: v for k, v in out.items() if v is not None}


def _trajectory(case, seed):
    """AR(1) chains with a common offset per chain: (samples, chains, dofs)."""
    g = _gen(seed)
    k, d, rho = case["chains"], case["dofs"], case["rho"]
    scale = torch.exp(-2.0 * torch.arange(d, device="cuda", dtype=torch.float64) / d)
    offset = 0.2 * _randn(g, k, d)
    e = _randn(g, case["samples"], k, d)
    x, rows = _randn(g, k, d), []
    for j in range(case["samples"]):
        x = rho * x + math.sqrt(1.0 - rho * rho) * e[j]
        rows.append((x + offset) * scale)
    return torch.stack(rows)


def _exact_diag(case, seed):
    X = _trajectory(case, seed).permute(2, 1, 0).contiguous()     # dof, chain, sample
    d, k, n = X.shape
    mean = X.mean(-1, keepdim=True)
    Xc = X - mean
    mk = mean[..., 0] - mean[..., 0].mean(-1, keepdim=True)
    W = torch.einsum("aks,bks->ab", Xc, Xc) / (k * (n - 1))
    V = (n - 1) / n * W + (k + 1) / (k * (k - 1)) * (mk @ mk.T)
    w, v = torch.diagonal(W), torch.diagonal(V)
    total = torch.zeros(d, dtype=torch.float64, device="cuda")
    alive, any_pair = torch.ones_like(total, dtype=torch.bool), torch.zeros_like(total)

    def mact(t):
        ac = (Xc[..., :n - t] * Xc[..., t:]).sum((-1, -2)) / (n * k)
        return 1.0 - (w - ac) / v

    for t in range(0, n - 1, 2):
        pair = (torch.ones_like(total) if t == 0 else mact(t)) + mact(t + 1)
        alive = alive & (pair > 0)
        if not bool(alive.any()):
            break
        total = total + torch.where(alive, pair, torch.zeros_like(pair))
        any_pair = any_pair + alive
    ess = torch.where(any_pair > 0, 1.0 / (2.0 * total - 1.0), torch.ones_like(total))
    lam, Q = torch.linalg.eigh(W)
    Wh = (Q * torch.sqrt(torch.clamp(lam, min=0.0))) @ Q.T
    sig = torch.linalg.eigvalsh(Wh @ V @ Wh)
    tw, tv = torch.trace(W), torch.trace(V)
    s = torch.sort(ess).values
    return dict(ess=ess, ess_median=0.5 * (s[(d - 1) // 2] + s[d // 2]),
                msj=((X[..., 1:] - X[..., :-1]) ** 2).sum() / (k * (n - 1)),
                mpsrf_w=tw + tv - 2.0 * torch.sqrt(torch.clamp(sig, min=0.0)).sum(),
                trace_w=tw, trace_v=tv)


def exact(case, seed):
    if case["kind"] == "noalloc":
        g = _gen(seed)
        w = _widths(case)
        Ws, bs = _weights(w, g)
        f, ds = _forward(Ws, bs, case["act"], _randn(g, case["points"], w[0]))
        return dict(f=f, J=_jacobian(Ws, ds))
    if case["kind"] == "diag":
        return _exact_diag(case, seed)
    return _exact_chains(case, seed)
