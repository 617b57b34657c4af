"""Kernels of small pools started early against the same ones in plain order.

In a context that times its kernels an event stands between any two launches,
so that each starts when the one before it has ended; without, the short ones
are placed while it still runs.  Both must give the same bits: on every shape
of test_gpu_early_launch.py, and with delayed acceptance, where the prior draw
reads the accept flags that the geometry kernel ahead of it writes.  Pools on
both sides of the sizes at which launches and the draw change over.
"""
import numpy as np
import pytest

from helpers import gpu_setup, variant
from test_gpu_early_launch import SHAPES
from workloads import CONFIGS, SEED_CHAINS, surrogate_inputs

pytestmark = pytest.mark.gpu


def _chains(dino, w, C, delayed, flags):
    ctx = dino.dino_init(0, flags=flags)
    try:
        sid = gpu_setup(dino, ctx, w)
        if delayed:  # the surrogate's own map, a little off, of its own coordinates
            E, _ = dino.dino_read_basis(ctx, sid, w.r, w.N)
            inp = surrogate_inputs(w)
            rng = np.random.default_rng(3)
            W = [x * (1 + 0.02 * rng.standard_normal(x.shape)) for x in inp["Ws"]]
            dino.dino_set_true_model(ctx, sid, E_t=E, W=W, b=inp["bs"], activation=w.activation)
        pool = dino.dino_chains_create(ctx, sid, C, 0.002, SEED_CHAINS)
        dino.dino_chains_step(ctx, pool, 24, stats=False)
        out = dino.dino_chains_read(ctx, pool, C, w.r, w.N)
        out.update(dino.dino_chains_read_last(ctx, pool, C, w.r))
        if delayed:
            out.update(dino.dino_chains_read_da(ctx, pool, C))
        return out
    finally:
        ctx.close()


@pytest.mark.parametrize("C", [3, 152, 153, 609])
@pytest.mark.parametrize("shape,delayed", [(s, False) for s in SHAPES] +
                         [("fp64_r16", True), ("fp64_wb", True), ("bf16_wb", True),
                          ("bf16_rsized", True)])
def test_early_starts_change_no_bit(shape, delayed, C):
    import paper_2403_08220_gb300 as dino
    w = variant(CONFIGS["small_fp64"], **SHAPES[shape])
    early, plain = (_chains(dino, w, C, delayed, f) for f in (0, dino.DINO_FLAG_TIMING))
    moved = np.sum(plain["accepts"])
    assert 0 < moved
    if delayed:
        assert moved < 24 * C              # chains of both kinds in the same draw
    for k in plain:
        assert np.array_equal(np.asarray(early[k]), np.asarray(plain[k]), equal_nan=True), k
