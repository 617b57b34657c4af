"""FP64 products on the tensor cores where the operands' entries differ in scale.

Plain FP64 sums of products are accurate entry by entry: |error| <= K eps
sum_k |a_k b_k|, whatever the other outputs do with a large a_k.  The digit
products must be so too.  The surrogates here are linear (identity activation,
two layers), so that z = W0 x, f = W1 z and J = W1 W0 are the products
themselves, and the encode m_r = E m of an explicit basis is another.

Tolerance: 4 (K + 8) eps on the same sum of absolute values, for each product
of the chain (the reference is a plain FP64 product itself).
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

EPS = 2.0 ** -53


@pytest.fixture(scope="module")
def dino():
    import paper_2403_08220_gb300 as d
    return d


def _eval(dino, W, x, n_grid=17):
    r, dy = W[0].shape[1], W[1].shape[0]
    ctx = dino.dino_init(0)
    try:
        sid = dino.dino_load_surrogate(
            ctx, n_grid=n_grid, prior_gamma=0.1, prior_delta=1.0, r=r,
            widths=[r, W[0].shape[0], dy], activation=0, W=W, b=[np.zeros(w.shape[0]) for w in W],
            basis_kind=dino.DINO_BASIS_KLE, y=np.zeros(dy), noise_var=1.0,
            precision=dino.DINO_PREC_FP64, noise_map=dino.DINO_NOISE_CHOLESKY)
        return dino.dino_surrogate_eval(ctx, sid, x, dy, want_L=False)
    finally:
        ctx.close()


def _check(out, W, x):
    h, r = W[0].shape
    a0, a1 = np.abs(W[0]), np.abs(W[1])
    f, fs = (x @ W[0].T) @ W[1].T, (np.abs(x) @ a0.T) @ a1.T
    J, Js = W[1] @ W[0], a1 @ a0
    assert np.all(np.abs(out["f"] - f) <= 4 * (h + r + 16) * EPS * fs)
    assert np.all(np.abs(out["J"] - J[None]) <= 4 * (h + 8) * EPS * Js[None])


@pytest.mark.parametrize("size", [1e3, 1e6, 1e10, 1e18, 1e300])
@pytest.mark.parametrize("r,h,dy", [(130, 200, 129), (200, 400, 100), (64, 513, 40)])
def test_large_entry_in_a_column_of_zeros(dino, r, h, dy, size):
    rng = np.random.default_rng(11)
    W = [rng.standard_normal((h, r)), rng.standard_normal((dy, h))]
    W[0][:, 5] = 0.0                       # an input that nothing uses
    W[1][:, 9] = size                      # a hidden unit that no input reaches
    W[0][9, :] = 0.0
    x = rng.standard_normal((3, r))
    x[:, 5] = size
    _check(_eval(dino, W, x), W, x)


@pytest.mark.parametrize("precision", ["fp64", "bf16"])
def test_encode_of_a_field_with_filler_outside_the_basis(dino, precision):
    """Nodes that E does not read hold a large filler value."""
    rng = np.random.default_rng(12)
    n, r, C = 33, 40, 5
    N = n * n
    seen = np.flatnonzero(rng.random(N) < 0.6)
    Q, _ = np.linalg.qr(rng.standard_normal((len(seen), r)))
    E, D = np.zeros((r, N)), np.zeros((N, r))
    E[:, seen], D[seen] = Q.T, Q
    m0 = rng.standard_normal((C, N))
    m0[:, np.setdiff1d(np.arange(N), seen)] = 1e12
    widths = [r, 48, 33]
    W = [rng.standard_normal((o, i)) / np.sqrt(i) for i, o in zip(widths[:-1], widths[1:])]
    ctx = dino.dino_init(0)
    try:
        sid = dino.dino_load_surrogate(
            ctx, n_grid=n, prior_gamma=0.1, prior_delta=1.0, r=r, widths=widths, activation=1,
            W=W, b=[np.zeros(o) for o in widths[1:]], basis_kind=dino.DINO_BASIS_EXPLICIT, E=E,
            D=D, y=np.zeros(widths[-1]), noise_var=1.0,
            precision=dino.DINO_PREC_FP64 if precision == "fp64" else dino.DINO_PREC_BF16)
        pool = dino.dino_chains_create(ctx, sid, C, 0.01, 7, m0=m0)
        m_r = dino.dino_chains_read(ctx, pool, C, r, N, field=False)["m_r"]
    finally:
        ctx.close()
    used = m0[:, seen]
    assert np.all(np.abs(m_r - used @ Q) <= 4 * (N + 8) * EPS * (np.abs(used) @ np.abs(Q)))


def test_a_row_that_is_not_finite_reaches_every_product_with_it(dino):
    """A Jacobian column that overflows makes its row and column of J^T J not
    finite, as in plain arithmetic, and with them every eigenvalue of the
    derivative-informed basis: no pair may come out as if the column were zero."""
    rng = np.random.default_rng(13)
    r, h, dy, n = 140, 150, 30, 20
    W = [rng.standard_normal((h, r)), 1e10 * rng.standard_normal((dy, h))]
    W[0][:, 77] = 1e300
    ctx = dino.dino_init(0)
    try:
        sid = dino.dino_load_surrogate(
            ctx, n_grid=17, prior_gamma=0.1, prior_delta=1.0, r=r, widths=[r, h, dy], activation=0,
            W=W, b=[np.zeros(h), np.zeros(dy)], basis_kind=dino.DINO_BASIS_KLE, y=np.zeros(dy),
            noise_var=1.0, precision=dino.DINO_PREC_FP64)
        out = dino.dino_dis_from_surrogate(ctx, sid, n, 5, 8, r, 17 * 17)
    finally:
        ctx.close()
    assert not np.any(np.isfinite(out["eigvals"]))


# Pairs of outputs and inputs whose large entries do not meet: (what, W0, W1, x) of
# r inputs, h hidden units, dy outputs.


def _one_large_input(rng, r, h, dy, size):
    W = [rng.standard_normal((h, r)), rng.standard_normal((dy, h))]
    W[0][::2, 3] = 0.0                     # half of the units ignore the large input
    W[1][::3, 8] = 0.0
    W[1][:, 8] *= size
    x = rng.standard_normal((3, r))
    x[:, 3] = size
    return W, x


def _blocks(rng, r, h, dy, size):
    W = [rng.standard_normal((h, r)), rng.standard_normal((dy, h))]
    W[0][: h // 2, r // 2:] = 0.0          # two groups of inputs, three of units
    W[0][h // 2: h // 2 + 9, : r // 2] = 0.0
    W[1][: dy // 2, : h // 2] = 0.0
    W[0][: h // 2] *= size
    x = rng.standard_normal((3, r))
    x[:, : r // 2] *= size
    return W, x


def _pruned(rng, r, h, dy, size):
    W = [rng.standard_normal((h, r)) * (rng.random((h, r)) < 0.05),
         rng.standard_normal((dy, h)) * (rng.random((dy, h)) < 0.05)]
    x = rng.standard_normal((3, r)) * size ** rng.uniform(-1, 1, (3, r))
    return W, x


def _all_scales(rng, r, h, dy, size):
    s = lambda *n: rng.standard_normal(n) * size ** rng.uniform(-1, 1, n)
    return [s(h, r), s(dy, h)], s(3, r)


def _selection(rng, r, h, dy, size):
    W = [np.zeros((h, r)), np.zeros((dy, h))]
    W[0][np.arange(h), rng.integers(0, r, h)] = 1.0
    W[1][np.arange(dy), rng.integers(0, h, dy)] = 1.0
    return W, rng.standard_normal((3, r)) * size ** rng.uniform(-1, 1, (3, r))


@pytest.mark.parametrize("size", [1e2, 1e6, 1e9, 1e40])
@pytest.mark.parametrize("make", [_one_large_input, _blocks, _pruned, _all_scales, _selection])
@pytest.mark.parametrize("r,h,dy", [(130, 200, 129), (200, 400, 100), (65, 1030, 40),
                                    (40, 513, 200)])
def test_large_entries_that_meet_small_ones(dino, make, r, h, dy, size):
    W, x = make(np.random.default_rng(14), r, h, dy, size)
    _check(_eval(dino, W, x), W, x)


@pytest.mark.parametrize("tiny", [1e-308, 3e-310, 5e-324])
def test_subnormal_entries(dino, tiny):
    """Entries at the bottom of the range, alone in a row and beside others."""
    rng = np.random.default_rng(15)
    r, h, dy = 130, 200, 129
    W = [1e150 * rng.standard_normal((h, r)), rng.standard_normal((dy, h))]
    x = np.stack([np.full(r, tiny), np.where(np.arange(r) % 2, tiny, 1e-300),
                  np.where(np.arange(r) % 2, tiny, 1.0)])
    W[0][:60, ::2] = 0.0                   # units that see only the tiny entries
    out = _eval(dino, W, x)
    a0, a1 = np.abs(W[0]), np.abs(W[1])
    f, fs = (x @ W[0].T) @ W[1].T, (np.abs(x) @ a0.T) @ a1.T
    assert np.all(np.abs(out["f"] - f) <= 4 * (h + r + 16) * EPS * fs)
    W[0][:, 7] = 4 * tiny                  # a column of weights
    W[1][5] *= tiny                        # a row of them
    out = _eval(dino, W, np.ones((1, r)))
    J, Js = W[1] @ W[0], np.abs(W[1]) @ np.abs(W[0])
    assert np.all(np.abs(out["J"][0] - J) <= 4 * (h + 8) * (EPS * Js + 5e-324))
