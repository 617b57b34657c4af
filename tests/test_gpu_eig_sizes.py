"""The eigen map at the edges of its eigensolver, against the FP64 oracle.

d_y = 1 and 2 (one pair, none), both sides of each lane split (16/17 and
32/33) and the largest d_y = 64, odd and even, on the FP64 path at the FP64
parity bar; a hidden layer narrower than d_y gives M = I + K K^T repeated unit
eigenvalues.
"""
import numpy as np
import pytest

from helpers import (gpu_setup, oracle_chains, oracle_setup, rel_err, step_and_compare,
                     variant)
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


def test_data_so_precise_that_the_factor_leaves_the_range_of_fp32():
    """noise_var = 1e-42: the factored matrix has a diagonal of 1e40 and more.

    Such a posterior and one of noise_var = 1e-30 with the same data differ by
    1e-14 in the proposal and its mean, where I vanishes beside H = J^T J /
    noise_var, and by the factor 1e12 in log rho.
    """
    import paper_2403_08220_gb300 as dino

    C, outs = 5, []
    w = variant(CONFIGS["small_fp64"], n_grid=10, r=70, widths=[70, 41, 30, 20],
                basis_kind=BASIS_DIS, activation=1, noise_map="eigen")
    for noise_var in (1e-30, 1e-42):
        ctx = dino.dino_init(0)
        try:
            sid = gpu_setup(dino, ctx, w)
            dino.dino_set_data(ctx, sid, 0.1 * np.cos(np.arange(w.d_y)), noise_var)
            pool = dino.dino_chains_create(ctx, sid, C, 0.02, SEED_CHAINS)
            dino.dino_chains_step(ctx, pool, 1)
            out = dino.dino_chains_read_last(ctx, pool, C, w.r)
            out["log_rho"] = out["log_rho"] * noise_var
            out["phi"] = dino.dino_chains_read(ctx, pool, C, w.r, w.N)["phi"] * noise_var
            outs.append(out)
        finally:
            ctx.close()
    for k in ("b", "mu", "phi", "log_rho"):
        assert rel_err(outs[1][k], outs[0][k]) <= 1e-10, k
    assert np.array_equal(outs[1]["accepted"], outs[0]["accepted"])
