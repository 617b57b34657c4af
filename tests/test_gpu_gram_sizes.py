"""The r-sized path's I + J^T J / noise_var (tensor-core precision) at the edges
of its 64 x 64 blocks, 32-row stages and 64-row FP32 sums, r a multiple of 4
(16-byte copies) or not, factor in shared and in global memory.

The library's own FP32 Jacobian and factor L are read back: L L^T must be
I + J^T J / noise_var up to the FP32 rounding of sums of at most 64 products,
64 * 2^-24 of the same sum of absolute values (the double-float sums and the
factorisation are far below it).
"""
import numpy as np
import pytest

from workloads import mlp_weights

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("r,d_y", [
    (1, 1), (3, 5), (32, 63), (63, 64), (64, 65), (65, 31), (66, 129), (127, 96), (128, 200),
    (129, 32), (160, 33), (209, 70), (260, 301),
    # factors in global memory: the last 16-column panel with 16, 1 and 9 columns
    (239, 40), (240, 17), (600, 50),
])
def test_factor_of_the_librarys_own_jacobian(r, d_y):
    import paper_2403_08220_gb300 as dino

    widths = [r, 40, d_y]
    Ws, bs = mlp_weights(widths, r + d_y)
    ctx = dino.dino_init(0)
    try:
        sid = dino.dino_load_surrogate(
            ctx, n_grid=17 if r <= 289 else 25, prior_gamma=0.1, prior_delta=1.0, r=r, widths=widths, activation=1,
            W=Ws, b=bs, basis_kind=dino.DINO_BASIS_KLE, y=np.zeros(d_y), noise_var=0.37,
            precision=dino.DINO_PREC_BF16, noise_map=dino.DINO_NOISE_CHOLESKY)
        x = np.random.default_rng(1).standard_normal((3, r))
        o = dino.dino_surrogate_eval(ctx, sid, x, d_y)
    finally:
        ctx.close()
    for c in range(3):
        J, L = o["J"][c], o["L"][c]
        H = np.eye(r) + J.T @ J / 0.37
        bound = 64 * 2.0 ** -24 * (np.abs(J).T @ np.abs(J)) / 0.37 + 1e-12 * np.abs(H).max()
        assert np.all(np.abs(np.tril(L @ L.T - H)) <= bound), (r, d_y)
        g = J.T @ o["f"][c] / 0.37
        assert np.max(np.abs(o["g"][c] - g)) <= 1e-12 * np.max(np.abs(J).T @ np.abs(o["f"][c]) / 0.37)
        hld = np.sum(np.log(np.diag(L)))
        assert abs(o["hld"][c] - hld) <= 1e-11 * max(1.0, abs(hld))
