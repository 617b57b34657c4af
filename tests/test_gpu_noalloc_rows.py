"""The allocation-free Jacobian's row split and its chunks of points.

Rows per CTA with a remainder, one row per CTA, fewer rows than SMs, more
points than the fixed scratch holds slabs for (d_y = 1 and many layers: the
call runs in several chunks), against the FP64 oracle at the FP64 parity bar.
"""
import numpy as np
import pytest

from helpers import rel_err
from oracle import mlp
from workloads import mlp_weights

pytestmark = pytest.mark.gpu

TOL = 1e-10


@pytest.mark.parametrize("widths,act,n", [
    ([33, 41, 100], mlp.ACT_TANH, 1),
    ([200, 400, 400, 101], mlp.ACT_GELU, 11),
    ([7, 64, 200, 3, 90, 128], mlp.ACT_GELU, 20),
    ([5] + [100] * 10 + [1], mlp.ACT_TANH, 5242),
    ([12, 6000, 2], mlp.ACT_GELU, 40),
])
def test_rows_and_chunks(widths, act, n):
    torch = pytest.importorskip("torch")
    import paper_2403_08220_gb300 as dino

    Ws, bs = mlp_weights(widths, 17)
    dev = torch.device("cuda", 0)
    Wt = [torch.tensor(W, dtype=torch.float64, device=dev).contiguous() for W in Ws]
    bt = [torch.tensor(b, dtype=torch.float64, device=dev).contiguous() for b in bs]
    x = np.random.default_rng(3).standard_normal((n, widths[0]))
    f_ref, zs = mlp.forward(Ws, bs, act, x)
    J_ref = mlp.jacobian_reverse(Ws, act, zs)
    xt = torch.tensor(x, dtype=torch.float64, device=dev)
    ft = torch.full((n, widths[-1]), float("nan"), dtype=torch.float64, device=dev)
    Jt = torch.full((n, widths[-1], widths[0]), float("nan"), dtype=torch.float64, device=dev)
    dino.dino_surrogate_jacobian_noalloc(
        n, widths, act, [t.data_ptr() for t in Wt], [t.data_ptr() for t in bt], xt.data_ptr(),
        ft.data_ptr(), Jt.data_ptr(), torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    assert rel_err(ft.cpu().numpy(), f_ref) <= TOL
    assert rel_err(Jt.cpu().numpy(), J_ref) <= TOL


def test_host_threads_share_a_stream():
    """Calls of several threads on one stream: two networks, different numbers of
    points (and so of rows per CTA and shared memory); every call's own results."""
    torch = pytest.importorskip("torch")
    import threading

    import paper_2403_08220_gb300 as dino

    dev = torch.device("cuda", 0)
    st = torch.cuda.current_stream().cuda_stream
    jobs = []
    for k, (widths, n) in enumerate([([200, 400, 400, 100], 1), ([200, 400, 400, 100], 12),
                                     ([30, 900, 70], 8), ([30, 900, 70], 2)]):
        Ws, bs = mlp_weights(widths, 21 + k)
        x = np.random.default_rng(k).standard_normal((n, widths[0]))
        f_ref, zs = mlp.forward(Ws, bs, mlp.ACT_TANH, x)
        t = lambda a: torch.tensor(a, dtype=torch.float64, device=dev).contiguous()
        jobs.append(dict(widths=widths, n=n, W=[t(a) for a in Ws], b=[t(a) for a in bs], x=t(x),
                         f=t(np.full((20, n, widths[-1]), np.nan)),
                         J=t(np.full((20, n, widths[-1], widths[0]), np.nan)), f_ref=f_ref,
                         J_ref=mlp.jacobian_reverse(Ws, mlp.ACT_TANH, zs)))
    torch.cuda.synchronize()
    failed = []

    def work(j):
        try:
            for i in range(20):
                dino.dino_surrogate_jacobian_noalloc(
                    j["n"], j["widths"], mlp.ACT_TANH, [a.data_ptr() for a in j["W"]],
                    [a.data_ptr() for a in j["b"]], j["x"].data_ptr(), j["f"][i].data_ptr(),
                    j["J"][i].data_ptr(), st)
        except Exception as e:
            failed.append(e)

    threads = [threading.Thread(target=work, args=(j,)) for j in jobs]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    assert not failed
    for j in jobs:
        for i in range(20):
            assert rel_err(j["f"][i].cpu().numpy(), j["f_ref"]) <= TOL
            assert rel_err(j["J"][i].cpu().numpy(), j["J_ref"]) <= TOL


@pytest.mark.parametrize("widths,act,n", [
    ([20, 9], mlp.ACT_TANH, 700),                    # a CTA per point: one layer,
    ([3, 4, 2], mlp.ACT_GELU, 3000),                 # a small network,
    ([16, 64, 64, 49], mlp.ACT_GELU, 48),            # many points;
    ([16, 64, 64, 49], mlp.ACT_GELU, 24),            # rows over all SMs: fewer,
    ([16, 64, 64, 49], mlp.ACT_IDENTITY, 90),        # cheaper activations,
    ([20, 6000, 6000, 1], mlp.ACT_TANH, 60),         # more points than scratch slabs
])
def test_both_ways_of_taking_the_points(widths, act, n):
    """... a CTA per point, or every point's outputs over all SMs."""
    test_rows_and_chunks(widths, act, n)
