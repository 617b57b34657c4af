"""Diagnostics at the edges of their kernels, against the FP64 oracle.

Jacobi blocks of one, two and four columns with odd numbers of them, the
staged and unstaged autocorrelation kernel, lag passes that end inside their
eight lags or at the last sample, covariances with fewer samples than degrees
of freedom (a positive semidefinite W), a degree of freedom that never moves,
and the Gram matrix on the tensor cores (d >= 32).  Tolerances as in
test_gpu_diag.py: 1e-9 relative for the effective sample sizes and 1e-9 of
Tr V for the MPSRF, whose square roots turn a rounding error eps of a zero
eigenvalue into sqrt(eps) = 1.5e-8 of its scale: 2e-8 where W is singular.
"""
import numpy as np
import pytest

from oracle import diagnostics as dg

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dino():
    import paper_2403_08220_gb300 as d
    return d


@pytest.mark.parametrize("n_c,n_s,d,rho", [
    (2, 2, 1, 0.0),
    (3, 9, 2, 0.3),
    (5, 64, 7, 0.9),
    (4, 3000, 33, 0.99),       # long memory; 96 KB of staged samples
    (7, 4100, 5, 0.5),         # 230 KB of samples: not staged
    (10, 130, 305, 0.6),       # blocks of two columns, an odd number of blocks
    (6, 20, 40, 0.5),          # fewer samples than degrees of freedom
    (12, 160, 613, 0.4),       # blocks of four columns
])
def test_sizes(dino, n_c, n_s, d, rho):
    rng = np.random.default_rng(n_c + d)
    X = np.empty((n_c, n_s, d))
    x = rng.standard_normal((n_c, d))
    for j in range(n_s):
        x = rho * x + np.sqrt(1 - rho ** 2) * rng.standard_normal((n_c, d))
        X[:, j] = x + 0.3 * np.arange(n_c)[:, None] / n_c
    X *= np.exp(-3.0 * np.arange(d) / d)
    ctx = dino.dino_init(0)
    try:
        g = dino.dino_diag_create(ctx, n_c, d, n_s)
        for j in range(n_s):
            dino.dino_diag_push(ctx, g, X[:, j, :])
        out = dino.dino_diag_compute(ctx, g, d, mpsrf=True)
    finally:
        ctx.close()
    ess = dg.ess_fractions(X)
    W, V = dg.covariance_estimators(X)
    singular = n_c * (n_s - 1) < d + 5
    assert np.max(np.abs(out["ess"] - ess) / np.abs(ess)) <= 1e-9
    assert abs(out["msj"] - dg.mean_squared_jump(X)) <= 1e-12 * dg.mean_squared_jump(X)
    assert abs(out["trace_w"] - np.trace(W)) <= 1e-12 * np.trace(W)
    assert abs(out["trace_v"] - np.trace(V)) <= 1e-12 * np.trace(V)
    tol = (2e-8 * np.sqrt(d) if singular else 1e-9) * np.trace(V)
    assert abs(out["mpsrf_w"] - dg.wasserstein_mpsrf(W, V)) <= tol


def test_a_still_degree_of_freedom_and_repeated_columns(dino):
    """A zero column of W and exactly dependent ones: no NaN, the oracle's MPSRF."""
    rng = np.random.default_rng(4)
    n_c, n_s, d = 4, 50, 36
    X = rng.standard_normal((n_c, n_s, d)) + 0.2 * rng.standard_normal((n_c, 1, d))
    X[:, :, 5] = X[:, :, 9]
    X[:, :, 20] = 2.0 * X[:, :, 1] - X[:, :, 30]
    X[:, :, 11] = 1.5
    ctx = dino.dino_init(0)
    try:
        g = dino.dino_diag_create(ctx, n_c, d, n_s)
        for j in range(n_s):
            dino.dino_diag_push(ctx, g, X[:, j, :])
        out = dino.dino_diag_compute(ctx, g, d, mpsrf=True)
    finally:
        ctx.close()
    W, V = dg.covariance_estimators(X)
    assert abs(out["mpsrf_w"] - dg.wasserstein_mpsrf(W, V)) <= 2e-8 * 6 * np.trace(V)


def test_a_nan_sample_stays_in_its_degree_of_freedom(dino):
    """One NaN among d = 40 (Gram matrix on the tensor cores): the other degrees
    of freedom keep their bits, traces and MPSRF are NaN, as in plain arithmetic."""
    rng = np.random.default_rng(9)
    n_c, n_s, d = 3, 40, 40
    X = rng.standard_normal((n_c, n_s, d))
    res = []
    for bad in (False, True):
        if bad:
            X[1, 7, 5] = np.nan
        ctx = dino.dino_init(0)
        try:
            g = dino.dino_diag_create(ctx, n_c, d, n_s)
            for j in range(n_s):
                dino.dino_diag_push(ctx, g, X[:, j, :])
            res.append(dino.dino_diag_compute(ctx, g, d, mpsrf=True))
        finally:
            ctx.close()
    keep = np.arange(d) != 5
    assert np.array_equal(res[0]["ess"][keep], res[1]["ess"][keep])
    for k in ("msj", "trace_w", "trace_v", "mpsrf_w"):
        assert np.isfinite(res[0][k]) and np.isnan(res[1][k]), k


@pytest.mark.parametrize("d,span,polar", [
    (7, 2.0, False), (8, 2.0, True), (9, 4.0, True),   # from d = 8 on the polar factor
    (61, 6.0, True), (257, 1.0, True), (512, 1.0, True), (513, 1.0, False),
    (64, 26.0, False),    # scales down to 5e-12: the iteration gives up, Jacobi solves
])
def test_nuclear_norm_by_polar_factor_or_jacobi(dino, d, span, polar):
    rng = np.random.default_rng(d)
    n_c, n_s = 4, max(24, d)
    X = rng.standard_normal((n_c, n_s, d)) + 0.3 * rng.standard_normal((n_c, 1, d))
    X *= np.exp(-span * np.arange(d) / d)
    ctx = dino.dino_init(0)
    try:
        g = dino.dino_diag_create(ctx, n_c, d, n_s)
        for j in range(n_s):
            dino.dino_diag_push(ctx, g, X[:, j, :])
        out = dino.dino_diag_compute(ctx, g, d, mpsrf=True)
    finally:
        ctx.close()
    W, V = dg.covariance_estimators(X)
    assert (out["jacobi_sweeps"] == 0) == polar
    tol = (1e-9 if span < 10 else 2e-8 * np.sqrt(d)) * np.trace(V)
    assert abs(out["mpsrf_w"] - dg.wasserstein_mpsrf(W, V)) <= tol


@pytest.mark.parametrize("d", [4, 7, 520])
def test_degrees_of_freedom_of_very_different_scales(dino, d):
    """Scales down to 1e-30, whose column pairs meet at angles below 1e-45: the
    sweeps reported are at most the sixty that there are, and the result is the
    oracle's for the others (what the small ones add is below 1e-23 of it)."""
    rng = np.random.default_rng(d)
    n_c, n_s = 4, max(40, d)
    X = rng.standard_normal((n_c, n_s, d)) + 0.3 * rng.standard_normal((n_c, 1, d))
    X *= 10.0 ** np.where(np.arange(d) % 2, -24.0 - 6.0 * np.arange(d) / d, 0.0)
    ctx = dino.dino_init(0)
    try:
        g = dino.dino_diag_create(ctx, n_c, d, n_s)
        for j in range(n_s):
            dino.dino_diag_push(ctx, g, X[:, j, :])
        out = dino.dino_diag_compute(ctx, g, d, mpsrf=True)
    finally:
        ctx.close()
    W, V = dg.covariance_estimators(X[:, :, ::2])
    assert abs(out["mpsrf_w"] - dg.wasserstein_mpsrf(W, V)) <= 1e-9 * np.trace(V)
    assert 1 <= out["jacobi_sweeps"] <= 60


@pytest.mark.parametrize("d", [4, 520])
def test_sweeps_end_with_degrees_of_freedom_of_very_different_scales(dino, d):
    """... and the solve ends by itself (exact angles: 3 and 22 sweeps, against 5
    and 13 on one scale) instead of turning the same pairs by nothing to the end."""
    rng = np.random.default_rng(d)
    n_c, n_s = 4, max(40, d)
    X = rng.standard_normal((n_c, n_s, d)) + 0.3 * rng.standard_normal((n_c, 1, d))
    X *= 10.0 ** np.where(np.arange(d) % 2, -24.0 - 6.0 * np.arange(d) / d, 0.0)
    ctx = dino.dino_init(0)
    try:
        g = dino.dino_diag_create(ctx, n_c, d, n_s)
        for j in range(n_s):
            dino.dino_diag_push(ctx, g, X[:, j, :])
        out = dino.dino_diag_compute(ctx, g, d, mpsrf=True)
    finally:
        ctx.close()
    assert 1 <= out["jacobi_sweeps"] < 60


def test_contexts_of_two_threads_with_different_sizes(dino):
    """Calls of different sizes side by side, each in a context of its own: every
    call succeeds and gives what it gives alone."""
    import threading

    runs, errors = {}, []

    def compute(key, n_c, n_s, d, times):
        try:
            rng = np.random.default_rng(d)
            X = rng.standard_normal((n_c, n_s, d))
            ctx = dino.dino_init(0)
            try:
                g = dino.dino_diag_create(ctx, n_c, d, n_s)
                for j in range(n_s):
                    dino.dino_diag_push(ctx, g, X[:, j, :])
                runs[key] = [dino.dino_diag_compute(ctx, g, d, mpsrf=True) for _ in range(times)]
            finally:
                ctx.close()
        except Exception as e:
            errors.append(e)

    sizes = [(2, 2000, 40), (3, 60, 5), (2, 900, 300)]
    for i, s in enumerate(sizes):
        compute(("alone", i), *s, 1)
    threads = [threading.Thread(target=compute, args=(i, *s, 60)) for i, s in enumerate(sizes)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors
    for i in range(len(sizes)):
        ref = runs["alone", i][0]
        for out in runs[i]:
            assert np.array_equal(out["ess"], ref["ess"]) and out["mpsrf_w"] == ref["mpsrf_w"]
