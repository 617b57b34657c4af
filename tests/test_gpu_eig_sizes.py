"""The eigen map at the edges of its eigensolver, against the FP64 oracle.

d_y = 1 and 2 (one pair, none), both sides of each lane split (16/17 and
32/33) and the largest d_y = 64, odd and even, on the FP64 path at the FP64
parity bar; a hidden layer narrower than d_y gives M = I + K K^T repeated unit
eigenvalues.
"""
import pytest

from helpers import gpu_setup, oracle_chains, oracle_setup, step_and_compare, variant
from workloads import BASIS_DIS, CONFIGS, SEED_CHAINS

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d_y", [1, 2, 3, 15, 16, 17, 32, 33, 64])
def test_eigen_map_sizes(d_y):
    import paper_2403_08220_gb300 as dino

    w = variant(CONFIGS["small_fp64"], n_grid=10, r=70, widths=[70, 41, 30, d_y],
                basis_kind=BASIS_DIS, activation=1, noise_frac=0.2, noise_map="eigen")
    ctx = dino.dino_init(0)
    try:
        sid = gpu_setup(dino, ctx, w)
        sur, E, D = oracle_setup(w)
        C, dt = 7, 0.02
        pool = dino.dino_chains_create(ctx, sid, C, dt, SEED_CHAINS)
        och = oracle_chains(dino, ctx, sid, w, sur, E, D, C, dt)
        step_and_compare(dino, ctx, pool, och, w, C, 4, tol=1e-10)
    finally:
        ctx.close()
