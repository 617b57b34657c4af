"""Tensor-core Woodbury path over d_y: CTA sizes of the factor's and the
proposal's kernels (32/33, 64/65), several chains' Gram matrices in one 128-row
tile (128 / d_y of them, the last tile part-filled), against the FP64 oracle at
the path's bars (proposal and its mean to 1e-3 in the 2-norm per chain).
"""
import numpy as np
import pytest

from helpers import gpu_setup, oracle_chains, oracle_setup, variant
from workloads import BASIS_DIS, CONFIGS, SEED_CHAINS

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d_y", [1, 2, 9, 25, 31, 32, 33, 42, 43, 63, 64, 65, 127, 128])
def test_proposals_meet_the_bars(d_y):
    import paper_2403_08220_gb300 as dino

    w = variant(CONFIGS["small_fp64"], n_grid=13, r=140, widths=[140, 150, 145, d_y],
                basis_kind=BASIS_DIS, activation=2, noise_frac=0.1, precision="bf16",
                noise_map="perturbation")
    ctx = dino.dino_init(0)
    try:
        sid = gpu_setup(dino, ctx, w)
        sur, E, D = oracle_setup(w)
        C, dt = 11, 0.1
        pool = dino.dino_chains_create(ctx, sid, C, dt, SEED_CHAINS)
        och = oracle_chains(dino, ctx, sid, w, sur, E, D, C, dt)
        dino.dino_chains_step(ctx, pool, 1, stats=False)
        och.step()
        last = dino.dino_chains_read_last(ctx, pool, C, w.r)
        for k in ("mu", "b"):
            err = np.linalg.norm(last[k] - och.last[k], axis=1) / np.linalg.norm(
                och.last[k], axis=1)
            assert err.max() <= 1e-3, (k, err.max())
        # a chain's results do not depend on its place in a tile
        solo = dino.dino_chains_create(ctx, sid, 1, dt, SEED_CHAINS, chain_id_base=C - 1)
        dino.dino_chains_step(ctx, solo, 1, stats=False)
        one = dino.dino_chains_read_last(ctx, solo, 1, w.r)
        for k in ("mu", "b", "log_rho"):
            assert np.array_equal(one[k][0], last[k][C - 1]), k
    finally:
        ctx.close()


@pytest.mark.parametrize("d_y,r", [(129, 200), (150, 163), (191, 250), (192, 193)])
def test_more_observations_than_a_tensor_core_gram_tile(d_y, r):
    """128 < d_y <= 192: the geometry kernel forms J J^T itself."""
    import paper_2403_08220_gb300 as dino

    w = variant(CONFIGS["small_fp64"], n_grid=17, r=r, widths=[r, 260, 255, d_y],
                basis_kind=BASIS_DIS, activation=2, noise_frac=0.1, precision="bf16",
                noise_map="perturbation")
    ctx = dino.dino_init(0)
    try:
        sid = gpu_setup(dino, ctx, w)
        sur, E, D = oracle_setup(w)
        C, dt = 11, 0.1
        pool = dino.dino_chains_create(ctx, sid, C, dt, SEED_CHAINS)
        och = oracle_chains(dino, ctx, sid, w, sur, E, D, C, dt)
        dino.dino_chains_step(ctx, pool, 1, stats=False)
        och.step()
        last = dino.dino_chains_read_last(ctx, pool, C, w.r)
        for k in ("mu", "b"):
            err = np.linalg.norm(last[k] - och.last[k], axis=1) / np.linalg.norm(
                och.last[k], axis=1)
            assert err.max() <= 1e-3, (k, err.max())
        assert np.all(np.isfinite(last["log_rho"]))
    finally:
        ctx.close()
