"""Batches of nothing but matrices that the fixed-point QR leaves to FP64 (a column twice, as in keyhole or
line-of-sight channels): every form of the FP64 kernels, its results by backward error (as in
test_gpu_qr.py), and that such matrices run side by side.

The time limit is a ratio on the same GPU: FP64 multiply-adds cost it some 10 times the fixed-point ones, and
every matrix runs twice, so 25 times an ordinary batch's time is not reached unless the matrices wait for one
another (then it is the number of matrices that wait in a row, 100 and more in these batches)."""

import numpy as np
import pytest

from paper_2002_09561_gb300 import mdx
from paper_2002_09561_gb300 import workload as wl

from test_gpu_qr import _check

pytestmark = pytest.mark.gpu

SIZES = [(4, 4, 20000), (8, 6, 3000), (16, 16, 500), (16, 16, 1100), (16, 16, 9000), (17, 17, 1500), (32, 32, 4000),
         (33, 30, 300), (40, 40, 700), (64, 48, 400), (100, 100, 304), (128, 100, 160)]


def _time(f):
    import torch

    f()
    ms = []
    for _ in range(3):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        f()
        b.record()
        torch.cuda.synchronize()
        ms.append(a.elapsed_time(b))
    return min(ms)


@pytest.mark.parametrize("N,M,B", SIZES)
def test_batches_of_dependent_columns(N, M, B):
    import torch

    w = wl.generate(8500 + N + M, B, N, M, 16, 10.0)
    H, y = w["H"].copy(), w["y"].copy()
    H[:, :, M - 2] = H[:, :, 0]
    ctx = mdx.Context(0, B, N, M)
    Ht, yt, plain = (torch.from_numpy(x).cuda() for x in (H, y, w["H"]))
    R, yb = mdx.qr(ctx, Ht, yt)
    R, yb = R.cpu().numpy(), yb.cpu().numpy()
    # the repeated column leaves rounding noise, or nothing: its diagonal entry may be 0
    assert np.all(np.abs(R[:, 2 * M - 4, 2 * M - 4]) <= 8 * M * 2.0 ** -53 * np.sqrt((H * H).sum((1, 2, 3))))
    d = np.diagonal(R, axis1=1, axis2=2)
    fixed = R.copy()
    i = np.arange(2 * M)
    fixed[:, i, i] = np.where(d == 0.0, 1e-300, d)  # (_check wants positive diagonals)
    _check(H, y, fixed, yb)
    assert _time(lambda: mdx.qr(ctx, Ht, yt)) < 25 * _time(lambda: mdx.qr(ctx, plain, yt))


@pytest.mark.parametrize("n,counts", [(8, (1400,)), (16, (900, 2000)), (40, (30,))])
def test_requests_with_dependent_columns(n, counts):
    """The gather form (requests of one size class) against the uniform batch: status, symbols, metrics."""
    import torch

    for B in counts:
        w = wl.generate(8600 + n + B, B, n, n, 4, 12.0)
        H, y = w["H"].copy(), w["y"].copy()
        some = np.arange(B) % 3 != 0
        H[some, :, 1] = H[some, :, 0]
        H[5, :, n - 1] = 0.0
        H, y, nv = (torch.from_numpy(x).cuda() for x in (H, y, w["noise_var"]))
        ctx = mdx.Context(0, B, n, n)
        sym, met, vst, _ = mdx.detect_kbest(ctx, mdx.make_params(n, n, 4, K=16), H, y, nv)
        reqs = mdx.make_requests(np.full(B, n), n, 4, mdx.MDX_ALGO_KBEST, K=16)
        s2, m2, v2, _ = mdx.detect_mixed(ctx, reqs, H.reshape(-1), y.reshape(-1), nv)
        assert torch.equal(vst, v2) and int(vst[5]) == mdx.MDX_V_SINGULAR
        live = (vst != mdx.MDX_V_SINGULAR).cpu().numpy()
        assert live[~some].all()
        assert torch.equal(s2.view(B, n)[~some], sym[~some]) and torch.equal(m2[~some], met[~some])
