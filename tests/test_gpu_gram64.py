"""FP64 Woodbury path: Gram matrices J J^T on the tensor cores, and the prior
draw's mirrored halves, against the FP64 oracle at the FP64 parity bar.

d_y on both sides of the rule (23 forms it in the geometry kernel), of the
column tiles (64/65) and of the row tiles (128/129), hidden layers just wide
enough for the scratch and wider; odd and even grids, smaller and larger than
one round of the draw's tiles.
"""
import numpy as np
import pytest

from helpers import gpu_setup, oracle_chains, oracle_setup, step_and_compare, variant
from workloads import BASIS_DIS, CONFIGS, SEED_CHAINS

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_grid,widths", [
    (9, [40, 41, 23]),
    (10, [40, 41, 24]),
    (17, [70, 90, 80, 65]),
    (16, [96, 104, 64]),
    (24, [140, 160, 128]),
    (33, [200, 201, 210, 129]),
    (20, [250, 300, 190]),
    (71, [36, 60, 30]),
])
def test_chains_match_oracle(n_grid, widths):
    import paper_2403_08220_gb300 as dino

    w = variant(CONFIGS["small_fp64"], n_grid=n_grid, r=widths[0], widths=widths,
                basis_kind=BASIS_DIS, activation=2, noise_frac=0.2, noise_map="perturbation")
    ctx = dino.dino_init(0)
    try:
        sid = gpu_setup(dino, ctx, w)
        sur, E, D = oracle_setup(w)
        C, dt = 5, 0.01
        pool = dino.dino_chains_create(ctx, sid, C, dt, SEED_CHAINS)
        och = oracle_chains(dino, ctx, sid, w, sur, E, D, C, dt)
        st = dino.dino_chains_read(ctx, pool, C, w.r, w.N)
        assert np.max(np.abs(st["m"] - och.m)) <= 1e-12       # the initial prior draw
        step_and_compare(dino, ctx, pool, och, w, C, 3, tol=1e-10)
    finally:
        ctx.close()
