"""The double-float factorisation with tensor-core trailing updates, against FP64.

Small-integer weights and the identity activation make J exact, so I + J^T J is
exact in FP32 and the factor of the r-sized path must agree with an FP64
Cholesky.  Sizes around the 8- and 16-column panels, the 16-row and 32-column
work items, and each place of the factor (shared memory with 128, 256 and 512
threads, global memory); columns of J scaled by powers of two spread the
diagonal over twelve binary orders.  The double-float entries carry 48 bits
relative to the diagonal, so L L^T must reproduce the matrix to 2^-44 n of
sqrt(M_ii M_jj) (one rounding per column, a factor 16 for the worst case); that
error E moves half log det by at most sum |M^-1| |E| / 2.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("r", [1, 7, 8, 9, 15, 16, 17, 23, 24, 31, 32, 33, 47, 64, 65, 100, 127,
                               130, 160, 195, 207, 209, 240, 255, 400])
def test_factor_reproduces_the_matrix(r):
    import paper_2403_08220_gb300 as dino

    rng = np.random.default_rng(r)
    h, dy = 30, r + 11
    W1 = rng.integers(-1, 2, size=(h, r)) * 2.0 ** rng.integers(-6, 7, size=r)
    W2 = rng.integers(-1, 2, size=(dy, h)).astype(float)
    n = int(np.ceil(np.sqrt(r))) + 1
    ctx = dino.dino_init(0)
    try:
        sid = dino.dino_load_surrogate(
            ctx, n_grid=n, prior_gamma=0.1, prior_delta=1.0, r=r, widths=[r, h, dy],
            activation=0, W=[W1, W2], b=[np.zeros(h), np.zeros(dy)],
            basis_kind=dino.DINO_BASIS_KLE, y=np.zeros(dy), noise_var=1.0,
            precision=dino.DINO_PREC_BF16, noise_map=dino.DINO_NOISE_CHOLESKY)
        o = dino.dino_surrogate_eval(ctx, sid, rng.standard_normal((2, r)), dy)
    finally:
        ctx.close()
    for c in range(2):
        J = o["J"][c]
        assert np.array_equal(J, W2 @ W1)
        M = np.eye(r) + J.T @ J
        s = np.sqrt(np.diag(M))
        L = o["L"][c].astype(np.longdouble)
        err = np.abs((L @ L.T).astype(np.float64) - M) / np.outer(s, s)
        assert err.max() <= 2.0 ** -44 * max(r, 4), err.max()
        ref = np.linalg.slogdet(M)[1] / 2
        tol = 2.0 ** -45 * max(r, 4) * np.sum(np.abs(np.linalg.inv(M)) * np.outer(s, s))
        assert abs(o["hld"][c] - ref) <= tol + 1e-13 * abs(ref)


@pytest.mark.parametrize("r,dy,precision", [(204, 187, "bf16"), (204, 224, "bf16"),
                                            (202, 690, "bf16"), (888, 40, "bf16"),
                                            (885, 140, "bf16"), (200, 3630, "fp64")])
def test_sizes_whose_shared_memory_ends_at_the_limit(r, dy, precision):
    """The blocked factorisation's digits, or the staged rows of J, would end within
    the last 304 bytes of a CTA's shared memory, which static variables hold."""
    import paper_2403_08220_gb300 as dino

    rng = np.random.default_rng(r)
    h = 16
    W = [rng.integers(-1, 2, size=(h, r)).astype(float),
         rng.integers(-1, 2, size=(dy, h)).astype(float)]
    n = int(np.ceil(np.sqrt(r))) + 1
    ctx = dino.dino_init(0)
    try:
        sid = dino.dino_load_surrogate(
            ctx, n_grid=n, prior_gamma=0.1, prior_delta=1.0, r=r, widths=[r, h, dy],
            activation=0, W=W, b=[np.zeros(h), np.zeros(dy)], basis_kind=dino.DINO_BASIS_KLE,
            y=np.zeros(dy), noise_var=64.0 * h * dy,
            precision=dino.DINO_PREC_BF16 if precision == "bf16" else dino.DINO_PREC_FP64,
            noise_map=dino.DINO_NOISE_CHOLESKY)
        o = dino.dino_surrogate_eval(ctx, sid, rng.standard_normal((1, r)), dy, want_L=False)
    finally:
        ctx.close()
    J = W[1] @ W[0]
    assert np.array_equal(o["J"][0], J)
    ref = np.linalg.slogdet(np.eye(r) + J.T @ J / (64.0 * h * dy))[1] / 2
    assert abs(o["hld"][0] - ref) <= 1e-9 * max(1.0, abs(ref))


@pytest.mark.parametrize("r", [106, 107, 108, 109, 133, 134, 135, 136, 157, 158, 159, 160, 203,
                               204])
def test_both_sides_of_the_rule_for_the_blocked_factorisation(r):
    """... by the CTAs an SM (d_y = r + 11)."""
    test_factor_reproduces_the_matrix(r)


@pytest.mark.parametrize("r,dy", [(887, 30), (895, 902), (1024, 40)])
def test_global_factor_beyond_the_panel_of_digits(r, dy):
    """The largest factors: the panel holds no digits (r from about 890)."""
    import paper_2403_08220_gb300 as dino

    rng = np.random.default_rng(r)
    h = 30
    W1 = rng.integers(-1, 2, size=(h, r)) * 2.0 ** rng.integers(-6, 7, size=r)
    W2 = rng.integers(-1, 2, size=(dy, h)).astype(float)
    ctx = dino.dino_init(0)
    try:
        sid = dino.dino_load_surrogate(
            ctx, n_grid=33, prior_gamma=0.1, prior_delta=1.0, r=r, widths=[r, h, dy],
            activation=0, W=[W1, W2], b=[np.zeros(h), np.zeros(dy)],
            basis_kind=dino.DINO_BASIS_KLE, y=np.zeros(dy), noise_var=1.0,
            precision=dino.DINO_PREC_BF16, noise_map=dino.DINO_NOISE_CHOLESKY)
        o = dino.dino_surrogate_eval(ctx, sid, rng.standard_normal((1, r)), dy)
    finally:
        ctx.close()
    J = o["J"][0]
    assert np.array_equal(J, W2 @ W1)
    M = np.eye(r) + J.T @ J
    s = np.sqrt(np.diag(M))
    L = o["L"][0]
    err = np.abs(L @ L.T - M) / np.outer(s, s)   # the product's own rounding is below r 2^-53
    assert err.max() <= (2.0 ** -44 + 2.0 ** -53) * r, err.max()
