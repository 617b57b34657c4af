"""FP64 products on the tensor cores (operands split into exact digits).

The surrogate's forward pass and Jacobian in the FP64 path, at widths around
the kernel's edges: output tiles of 64 and 32 columns, 32-column stages, the
512-column exact chunks, row tiles of 128, both Jacobian orders, weights that
leave an input unused or weigh it by 1e-8 (column exponents).  Reference: the
FP64 oracle.  Tolerance: every product of the chain is a sum of at most K
terms, so both sides differ by at most (K + 8) eps per product from the exact
value, measured against the same chain of absolute values (GELU's derivatives
and values add a few eps each): 4 * sum_l (K_l + 8) eps on that scale.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

EPS = 2.0 ** -53


@pytest.fixture(scope="module")
def dino():
    import paper_2403_08220_gb300 as d
    return d


def _load(dino, ctx, n_grid, widths, act, W, b):
    return dino.dino_load_surrogate(
        ctx, n_grid=n_grid, prior_gamma=0.1, prior_delta=1.0, r=widths[0], widths=widths,
        activation=act, W=W, b=b, basis_kind=dino.DINO_BASIS_KLE, y=np.zeros(widths[-1]),
        noise_var=1.0, precision=dino.DINO_PREC_FP64)


def _weights(widths, seed):
    rng = np.random.default_rng(seed)
    W = [rng.standard_normal((o, i)) / np.sqrt(i) for i, o in zip(widths[:-1], widths[1:])]
    return W, [0.1 * rng.standard_normal(o) for o in widths[1:]], rng


@pytest.mark.parametrize("widths,points,act", [
    ([130, 200, 129, 130], 1, 2),           # one point; ragged column tiles
    ([200, 400, 400, 100], 3, 2),           # two 128-row tiles and a remainder
    ([64, 513, 1030, 33], 2, 1),            # chunks of 512 columns and a remainder
    ([128, 256, 300, 200], 5, 2),           # forward-mode Jacobian
    ([140, 511, 512, 140, 131], 2, 2),      # a product between the first and the last
])
def test_forward_and_jacobian(dino, widths, points, act):
    from oracle import mlp
    W, b, rng = _weights(widths, 5)
    W[0][:, 3] *= 1e-8                      # an input that is hardly used, but large
    W[1][:, 7] = 0.0                        # a hidden unit that is not used at all
    x = rng.standard_normal((points, widths[0]))
    x[:, 3] *= 1e6
    ctx = dino.dino_init(0)
    try:
        sid = _load(dino, ctx, 33, widths, act, W, b)
        out = dino.dino_surrogate_eval(ctx, sid, x, widths[-1], want_L=False)
    finally:
        ctx.close()
    f, zs = mlp.forward(W, b, act, x)
    J = mlp.jacobian_reverse(W, act, zs)
    # the same chains of absolute values (|act(z)| <= |z| + 1, |act'| <= 1.13)
    a = np.abs(x)
    for Wl, bl in zip(W[:-1], b[:-1]):
        a = np.minimum(a @ np.abs(Wl).T + np.abs(bl), 1e3)
    fs = a @ np.abs(W[-1]).T + np.abs(b[-1])
    Js = np.abs(W[-1])
    for Wl in reversed(W[:-1]):
        Js = (1.13 * Js) @ np.abs(Wl)
    tol = 4 * sum(k + 8 for k in widths[:-1]) * EPS
    assert np.max(np.abs(out["f"] - f) / fs) < tol
    assert np.max(np.abs(out["J"] - J) / (Js + 1e-300)) < tol * 4  # act' moves by |act''| dz


def test_rows_with_infinities_and_nans_stay_alone(dino):
    """A NaN or an infinity reaches its own point only, as in a plain product."""
    widths = [160, 200, 150, 120]
    W, b, rng = _weights(widths, 6)
    x = rng.standard_normal((7, widths[0]))
    bad = x.copy()
    bad[1, 5] = np.nan
    bad[4, 0] = np.inf
    ctx = dino.dino_init(0)
    try:
        sid = _load(dino, ctx, 17, widths, 1, W, b)
        ref = dino.dino_surrogate_eval(ctx, sid, x, widths[-1], want_L=False)
        out = dino.dino_surrogate_eval(ctx, sid, bad, widths[-1], want_L=False)
    finally:
        ctx.close()
    ok = [0, 2, 3, 5, 6]
    for k in ("f", "J", "phi", "g", "hld"):
        assert np.array_equal(out[k][ok], ref[k][ok]), k
    assert np.all(np.isnan(out["f"][1])) and np.all(np.isnan(out["J"][1]))
    # tanh of an infinite pre-activation is +-1: the value stays finite, the Jacobian is 0
    z = W[0][:, 0]
    a = np.sign(z)
    f = np.tanh(W[1] @ a + b[1])
    assert np.allclose(out["f"][4], W[2] @ f + b[2], rtol=0, atol=1e-13)
    assert np.all(out["J"][4] == 0.0)


def test_points_do_not_depend_on_their_company(dino):
    """The same bits for a point alone and among others (row chunks, tiles)."""
    widths = [200, 400, 400, 100]
    W, b, rng = _weights(widths, 7)
    x = rng.standard_normal((70, widths[0]))
    ctx = dino.dino_init(0)
    try:
        sid = _load(dino, ctx, 33, widths, 2, W, b)
        many = dino.dino_surrogate_eval(ctx, sid, x, widths[-1], want_L=False)
        for k in (0, 37, 69):
            one = dino.dino_surrogate_eval(ctx, sid, x[k], widths[-1], want_L=False)
            for q in ("f", "J", "phi", "g"):
                assert np.array_equal(one[q][0], many[q][k]), (k, q)
    finally:
        ctx.close()


def test_more_hidden_units_than_a_grid_has_second_rows(dino):
    """600000 hidden units between 16 inputs and 2 outputs: small products (no
    digits) whose column tiles outnumber a grid's second dimension."""
    widths = [16, 600000, 2]
    W, b, rng = _weights(widths, 8)
    x = rng.standard_normal((2, 16))
    ctx = dino.dino_init(0)
    try:
        sid = _load(dino, ctx, 9, widths, 1, W, b)
        out = dino.dino_surrogate_eval(ctx, sid, x, 2, want_L=False)
    finally:
        ctx.close()
    z = x @ W[0].T + b[0]
    t = np.tanh(z)
    f = t @ W[1].T + b[1]
    J = np.einsum("ih,nh,hr->nir", W[1], 1 - t * t, W[0], optimize=True)
    # sums of 600000 terms of order 1/800: rounding errors of at most K eps of the
    # sum of their magnitudes
    tol = 4 * (600000 + 16) * EPS
    assert np.all(np.abs(out["f"] - f) <= tol * (np.abs(t) @ np.abs(W[1]).T + np.abs(b[1])))
    Js = np.einsum("ih,nh,hr->nir", np.abs(W[1]), 1 - t * t, np.abs(W[0]), optimize=True)
    assert np.all(np.abs(out["J"] - J) <= tol * Js)
