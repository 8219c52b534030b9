"""The QR's forms (several matrices per warp, one CTA per matrix, the FP64
form for matrices a fixed scale per column does not suit) at the edges of
their ranges, by backward error: R^H R = H^H H and R^H ybar = H^H y hold to
c n u ||H||^2 and c n u ||H|| ||y|| for any backward-stable QR (n reflectors of
relative error a few u each, u = 2^-53; c = 8)."""

import numpy as np
import pytest

from paper_2002_09561_gb300 import mdx
from paper_2002_09561_gb300 import workload as wl

pytestmark = pytest.mark.gpu
U = 2.0 ** -53


def _run(H, y):
    import torch

    B, N, M = H.shape[:3]
    ctx = mdx.Context(0, B, N, M)
    R, yb = mdx.qr(ctx, torch.from_numpy(H).cuda(), torch.from_numpy(y).cuda())
    return R.cpu().numpy(), yb.cpu().numpy()


def _check(H, y, R, yb, which=slice(None)):
    H, y, R, yb = H[which], y[which], R[which], yb[which]
    M = H.shape[2]
    Hc, yc = H[..., 0] + 1j * H[..., 1], y[..., 0] + 1j * y[..., 1]
    Rc = R[:, 0::2, 0::2] - 1j * R[:, 0::2, 1::2]
    ybc = yb[:, 0::2] + 1j * yb[:, 1::2]
    assert np.array_equal(R[:, 0::2, 0::2], R[:, 1::2, 1::2])
    assert np.array_equal(np.triu(R), R) and np.all(np.diagonal(Rc, axis1=1, axis2=2).real > 0)
    gh = lambda A: np.conj(np.swapaxes(A, 1, 2))  # noqa: E731
    nh = np.linalg.norm(Hc, axis=(1, 2))
    e = np.linalg.norm(gh(Rc) @ Rc - gh(Hc) @ Hc, axis=(1, 2)) / nh ** 2
    ey = np.linalg.norm((gh(Rc) @ ybc[..., None] - gh(Hc) @ yc[..., None])[..., 0], axis=1) / (
        nh * np.linalg.norm(yc, axis=1))
    assert e.max() < 8 * M * U and ey.max() < 8 * M * U, (e.max(), ey.max())


@pytest.mark.parametrize("N,M,B", [
    (1, 1, 3), (4, 4, 1217), (5, 2, 1218), (8, 8, 1217), (8, 7, 16385), (9, 9, 1219), (12, 9, 9729), (16, 16, 1216),
    (16, 16, 1223), (17, 3, 1825), (24, 24, 1826), (24, 23, 4865), (25, 25, 1827), (32, 32, 1824), (32, 32, 1829),
    (33, 33, 2), (47, 45, 609), (64, 64, 3), (81, 80, 2), (100, 100, 2), (128, 100, 2),
    (16, 16, 153), (31, 31, 152), (32, 32, 153), (48, 48, 152), (48, 48, 153), (49, 49, 1), (65, 64, 2), (96, 96, 2),
    (97, 97, 1), (128, 99, 2)])
def test_qr_forms_at_their_edges(N, M, B):
    w = wl.generate(8100 + N + B, B, N, M, 16, 10.0)
    _check(w["H"], w["y"], *_run(w["H"], w["y"]))


@pytest.mark.parametrize("N,M,B", [(4, 4, 1300), (16, 16, 1300), (24, 20, 2000), (16, 16, 8), (40, 40, 8)])
def test_matrices_left_to_the_fp64_form(N, M, B):
    """Nearly dependent columns, columns far apart in scale, scales near the ends of the fixed-point
    range, an exactly zero column, NaN: next to ordinary matrices, which must not change."""
    w = wl.generate(8200 + N, B, N, M, 16, 10.0)
    H, y = w["H"].copy(), w["y"].copy()
    plain, yplain = _run(H, y)
    H[1, :, 1] = H[1, :, 0] * (1 + 1e-9)       # a residual column of 1e-9
    H[2, :, 2] *= 1e-30
    H[3] *= 1e-150
    y[3] = 0.0
    H[4, :, M - 1] = 0.0
    H[5, 0, 0, 0] = np.nan
    R, yb = _run(H, y)
    keep = [0] + list(range(6, B))
    assert np.array_equal(R[keep], plain[keep]) and np.array_equal(yb[keep], yplain[keep])
    _check(H, y, R, yb, [0, 1, 2, 6, 7])
    assert np.all(yb[3] == 0.0)
    np.testing.assert_allclose(R[3] * 1e150, plain[3], rtol=0, atol=8 * M * U * np.linalg.norm(plain[3]) * 10)
    assert R[4, 2 * M - 1, 2 * M - 1] == 0.0 and np.isnan(R[5]).any()


def test_uneven_batch_uses_the_same_forms():
    """1,300 requests of one class (several matrices per warp in the gather form) detect as the uniform batch does."""
    import torch

    n, qam, B = 8, 16, 1300
    w = wl.generate(8300, B, n, n, qam, 14.0)
    H, y, nv = (torch.from_numpy(w[k]).cuda() for k in ("H", "y", "noise_var"))
    ctx = mdx.Context(0, B, n, n)
    uniform = mdx.detect_kbest(ctx, mdx.make_params(n, n, qam, K=16), H, y, nv)
    reqs = mdx.make_requests(np.full(B, n), n, qam, mdx.MDX_ALGO_KBEST, K=16)
    sym, met, _, _ = mdx.detect_mixed(ctx, reqs, H.reshape(-1), y.reshape(-1), nv)
    assert torch.equal(sym.view(B, n), uniform[0]) and torch.equal(met, uniform[1])


@pytest.mark.parametrize("N,M,B", [(8, 8, 1300), (16, 16, 1300), (20, 17, 2000), (16, 16, 4), (64, 50, 4)])
def test_zeros_stay_exactly_zero(N, M, B):
    """y = 0 gives ybar = 0 and a diagonal channel a diagonal R, exactly (ties between leaves are then
    exact ties), and the identity gives the identity."""
    w = wl.generate(8400 + N, B, N, M, 16, 10.0)
    H, y = w["H"].copy(), w["y"].copy()
    y[0] = 0.0
    H[1:3] = 0.0
    H[1, np.arange(M), np.arange(M), 0] = 1.0
    H[2, np.arange(M), np.arange(M), 0] = 1.0 + np.arange(M) / 7.0
    R, yb = _run(H, y)
    assert np.all(yb[0] == 0.0)
    assert np.array_equal(R[1], np.eye(2 * M))
    assert np.array_equal(R[2], np.diag(np.repeat(1.0 + np.arange(M) / 7.0, 2)))
