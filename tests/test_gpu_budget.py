"""The HBM budget and the digits of the FP64 products' weights.

The digits lie beside the budget: a surrogate takes what its FP64 arrays take,
a pool that fits with them loads, steps and evaluates with the same bits as in
a context without a limit, and one byte less is refused.
"""
import numpy as np
import pytest

from helpers import gpu_setup, variant
from workloads import BASIS_DIS, CONFIGS, SEED_CHAINS

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dino():
    import paper_2403_08220_gb300 as d
    return d


WIDTHS = [140, 150, 160, 130]


def _used(dino, ctx):
    return dino.dino_serve_status(ctx)["hbm_used"]


def test_budget_of_an_fp64_surrogate_and_its_pool(dino):
    w = variant(CONFIGS["small_fp64"], n_grid=17, r=WIDTHS[0], widths=WIDTHS,
                basis_kind=BASIS_DIS, activation=2, noise_frac=0.3)
    C, N = 9, w.N
    ctx = dino.dino_init(0)
    sid = gpu_setup(dino, ctx, w)
    base = _used(dino, ctx)
    entries = 2 * w.r * N + N + N + w.d_y        # E, D, the sine matrix, the spectrum, y
    entries += sum(2 * a * b + b for a, b in zip(WIDTHS[:-1], WIDTHS[1:]))
    assert base == 8 * entries
    pool = dino.dino_chains_create(ctx, sid, C, 0.002, SEED_CHAINS)
    pool_bytes = _used(dino, ctx) - base
    dino.dino_chains_step(ctx, pool, 3)
    ref = dino.dino_chains_read(ctx, pool, C, w.r, N)
    ctx.close()
    # gpu_setup holds a second surrogate for a while: no more than a pool
    for budget, fits in ((base + pool_bytes, True), (base + pool_bytes - 1, False)):
        ctx = dino.dino_init(0, hbm_budget_bytes=max(budget, 0))
        try:
            sid = gpu_setup(dino, ctx, w)
            if not fits:
                with pytest.raises(dino.DinoError) as e:
                    dino.dino_chains_create(ctx, sid, C, 0.002, SEED_CHAINS)
                assert e.value.code == dino.DINO_ENOMEM
                continue
            pool = dino.dino_chains_create(ctx, sid, C, 0.002, SEED_CHAINS)
            dino.dino_chains_step(ctx, pool, 3)
            out = dino.dino_chains_read(ctx, pool, C, w.r, N)
            for k in ref:
                assert np.array_equal(out[k], ref[k]), k
        finally:
            ctx.close()


def test_gram_products_within_the_budget(dino):
    """The diagnostics' digits count while the call lasts and are given back; where
    they do not fit the call still succeeds."""
    rng = np.random.default_rng(1)
    n_c, n_s, d = 4, 300, 60
    X = rng.standard_normal((n_c, n_s, d)) + 0.2 * rng.standard_normal((n_c, 1, d))
    outs = []
    tight = 0
    for _ in range(2):
        ctx = dino.dino_init(0, hbm_budget_bytes=tight)
        try:
            g = dino.dino_diag_create(ctx, n_c, d, n_s)
            for j in range(n_s):
                dino.dino_diag_push(ctx, g, X[:, j, :])
            base = _used(dino, ctx)
            outs.append(dino.dino_diag_compute(ctx, g, d, mpsrf=True))
            assert _used(dino, ctx) == base
            # the computation's own arrays, and a third of the digits
            tight = base + 8 * (d * n_c * n_s + d * n_c + 9 * d * d + d + 400) + 6 * d * n_c * n_s
        finally:
            ctx.close()
    assert np.array_equal(outs[0]["ess"], outs[1]["ess"])
    assert abs(outs[0]["mpsrf_w"] - outs[1]["mpsrf_w"]) <= 1e-11 * outs[0]["trace_v"]


@pytest.mark.parametrize("widths", [[40, 1500, 1500, 40], [36, 1500, 40, 900, 2],
                                    [32, 1200, 1100, 48]])
def test_one_point_where_a_buffer_holds_no_row_of_digits(dino, widths):
    """Wide layers between few inputs and outputs: one point's Jacobian (the scratch
    of the products in between) is smaller than the digits of one row.  The same
    bits as among others, whose buffers hold many."""
    rng = np.random.default_rng(2)
    W = [rng.standard_normal((o, i)) / np.sqrt(i) for i, o in zip(widths[:-1], widths[1:])]
    x = rng.standard_normal((60, widths[0]))
    ctx = dino.dino_init(0)
    try:
        sid = dino.dino_load_surrogate(
            ctx, n_grid=13, prior_gamma=0.1, prior_delta=1.0, r=widths[0], widths=widths,
            activation=2, W=W, b=[0.1 * rng.standard_normal(o) for o in widths[1:]],
            basis_kind=dino.DINO_BASIS_KLE, y=np.zeros(widths[-1]), noise_var=1.0)
        many = dino.dino_surrogate_eval(ctx, sid, x, widths[-1], want_L=False)
        for k in (0, 59):
            one = dino.dino_surrogate_eval(ctx, sid, x[k], widths[-1], want_L=False)
            for q in ("f", "J"):
                assert np.array_equal(one[q][0], many[q][k]), (k, q)
    finally:
        ctx.close()
