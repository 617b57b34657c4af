"""Kernels of small pools start before the ones ahead of them have ended; the
results must be those of transitions issued one at a time with the stream idle
between them (bit for bit: the same kernels on the same data).  Pools on both
sides of the sizes at which launches and the prior draw change over (152 and
608 CTAs), on the Woodbury path, the r-sized path and the eigen map, with
accepted moves, so that a field or factor read too early would show.
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


SHAPES = {
    "fp64_r16": dict(precision="fp64", noise_map="cholesky"),
    "fp64_wb": dict(precision="fp64", n_grid=13, r=40, widths=[40, 48, 17], basis_kind=BASIS_DIS,
                    activation=2, noise_frac=0.3),
    "bf16_wb": dict(precision="bf16", n_grid=33, r=64, widths=[64, 96, 96, 40],
                    basis_kind=BASIS_DIS, activation=2, noise_frac=0.3),
    "bf16_rsized": dict(precision="bf16", n_grid=33, r=40, widths=[40, 96, 64],
                        basis_kind=BASIS_DIS, activation=2, noise_frac=0.3),
    "bf16_eigen": dict(precision="bf16", n_grid=17, r=64, widths=[64, 96, 21],
                       basis_kind=BASIS_DIS, activation=2, noise_frac=0.3, noise_map="eigen"),
}


@pytest.mark.parametrize("C", [3, 152, 153, 609])
@pytest.mark.parametrize("shape", list(SHAPES))
def test_back_to_back_is_one_at_a_time(dino, shape, C):
    w = variant(CONFIGS["small_fp64"], **SHAPES[shape])
    ctx = dino.dino_init(0)
    try:
        sid = gpu_setup(dino, ctx, w)
        steps, dt = 24, 0.002
        together = dino.dino_chains_create(ctx, sid, C, dt, SEED_CHAINS)
        single = dino.dino_chains_create(ctx, sid, C, dt, SEED_CHAINS)
        dino.dino_chains_step(ctx, together, steps, stats=False)
        a = dino.dino_chains_read(ctx, together, C, w.r, w.N)
        la = dino.dino_chains_read_last(ctx, together, C, w.r)
        moved = 0
        for _ in range(steps):
            dino.dino_chains_step(ctx, single, 1, stats=False)
            moved += int(np.sum(dino.dino_chains_read_last(ctx, single, C, w.r)["accepted"]))
        b = dino.dino_chains_read(ctx, single, C, w.r, w.N)
        lb = dino.dino_chains_read_last(ctx, single, C, w.r)
    finally:
        ctx.close()
    assert moved > 0
    for x, y in ((a, b), (la, lb)):
        for k in x:
            assert np.array_equal(np.asarray(x[k]), np.asarray(y[k]), equal_nan=True), k
