"""FP64 products on the tensor cores do not depend on the pool: a chain alone and
among others gives the same bits where the pool's own buffers hold less than
one row of digits (few chains, few observations) and where they hold many.
"""
import numpy as np
import pytest

from helpers import gpu_setup, variant
from workloads import BASIS_DIS, CONFIGS, SEED_CHAINS

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp64", "bf16"])
@pytest.mark.parametrize("d_y", [1, 2, 4, 30])
def test_a_chain_alone_and_among_others(precision, d_y):
    import paper_2403_08220_gb300 as dino

    w = variant(CONFIGS["small_fp64"], n_grid=20, r=140, widths=[140, 300, 160, 145, d_y],
                basis_kind=BASIS_DIS, activation=2, noise_frac=0.1, precision=precision)
    ctx = dino.dino_init(0)
    try:
        sid = gpu_setup(dino, ctx, w)
        C, dt, res = 11, 0.05, []
        for base, n in ((0, C), (C - 1, 1)):
            p = dino.dino_chains_create(ctx, sid, n, dt, SEED_CHAINS, chain_id_base=base)
            dino.dino_chains_step(ctx, p, 2, stats=False)
            o = dino.dino_chains_read(ctx, p, n, w.r, w.N)
            o.update(dino.dino_chains_read_last(ctx, p, n, w.r))
            res.append({k: v[-1] for k, v in o.items()})
        for k in res[0]:
            if k != "m" or precision == "fp64":  # BF16: the complement splits K by pool size
                assert np.array_equal(res[0][k], res[1][k]), k
    finally:
        ctx.close()
