"""The QR on receive antennas of very different scale, strongest first (pre-whitened or attenuated rows):
row-wise accuracy of R and ybar, which FP64 Householder reflections keep for such an order of the rows and a
fixed scale per column does not; and received vectors of subnormal numbers.

Bound: every row of R and ybar goes through at most M reflectors, each with a relative error of a few u of
that row (u = 2^-53), so the root mean square of the rows' relative errors is held to 8 M u, the constant of
test_gpu_qr.py.  A fixed scale per column gives 2^-58 of the column's norm instead, 2^20 times that of a
row graded down to 1e-6."""

import numpy as np
import pytest

from paper_2002_09561_gb300 import workload as wl

from test_gpu_qr import U, _check, _run

pytestmark = pytest.mark.gpu


def _householder(H, y):
    """Complex R and ybar in extended precision."""
    A = np.concatenate([H[..., 0] + 1j * H[..., 1], (y[..., 0] + 1j * y[..., 1])[..., None]], 2).astype(np.clongdouble)
    M = H.shape[2]
    for k in range(M):
        x = A[:, k:, k].copy()
        s = np.sqrt((x.real ** 2 + x.imag ** 2).sum(1))
        ph = x[:, 0] / np.abs(x[:, 0])
        x[:, 0] += ph * s
        w = (x.conj()[:, :, None] * A[:, k:, k:]).sum(1) * (2 / (x.real ** 2 + x.imag ** 2).sum(1))[:, None]
        A[:, k:, k:] -= x[:, :, None] * w[:, None, :]
        A[:, k] *= -ph.conj()[:, None]
    return np.triu(A[:, :M, :M]), A[:, :M, M]


def _row_errors(H, y, R, yb):
    ref, yref = _householder(H, y)
    Rc = R[:, 0::2, 0::2] - 1j * R[:, 0::2, 1::2]
    ybc = yb[:, 0::2] + 1j * yb[:, 1::2]
    eR = np.sqrt((np.abs(Rc - ref) ** 2).sum(2) / (np.abs(ref) ** 2).sum(2)).astype(float)
    ey = (np.abs(ybc - yref) / np.abs(yref)).astype(float)
    return eR, ey


@pytest.mark.parametrize("N,M,copies", [(2, 2, 1), (4, 4, 200), (8, 8, 1), (8, 8, 200), (16, 12, 1), (16, 16, 200),
                                        (24, 24, 300), (32, 32, 1), (40, 40, 1), (64, 50, 1)])
@pytest.mark.parametrize("down", [1e-3, 1e-6, 1e-12])
def test_rows_graded_down_keep_their_accuracy(N, M, copies, down):
    w = wl.generate(8700 + N + M, 8, N, M, 16, 10.0)
    scale = down ** (np.arange(N) / (N - 1))
    H, y = w["H"] * scale[:, None, None], w["y"] * scale[:, None]
    R, yb = _run(np.concatenate([H] * copies), np.concatenate([y] * copies))
    assert all(np.array_equal(R[:8], R[8 * c:8 * c + 8]) for c in range(copies))
    eR, ey = _row_errors(H, y, R[:8], yb[:8])
    assert np.sqrt((eR ** 2).mean()) < 8 * M * U
    # ybar: rows that happen to cancel are small themselves, so their median stands for the rows
    assert np.median(ey) < 8 * M * U


@pytest.mark.parametrize("N,M", [(8, 8), (16, 10), (40, 40)])
def test_zero_rows_and_other_orders_are_ordinary(N, M):
    """Zero rows (padding), small rows anywhere but last, columns of very different power: backward error."""
    w = wl.generate(8800 + N, 6, N, M, 16, 10.0)
    H, y = w["H"].copy(), w["y"].copy()
    H[1, 2] = 0.0
    H[2, N // 2] *= 1e-9
    H[3] *= np.geomspace(1e-6, 1.0, N)[:, None, None]
    H[4] *= np.geomspace(1.0, 1e-6, M)[None, :, None]
    if N > M:
        H[5, M:] = 0.0
    _check(H, y, *_run(H, y))


@pytest.mark.parametrize("N,M,B", [(4, 4, 2), (16, 16, 1300), (40, 40, 2)])
def test_subnormal_received_vectors(N, M, B):
    w = wl.generate(8900 + N, B, N, M, 16, 10.0)
    H, y = w["H"], w["y"].copy()
    _, plain = _run(H, y)
    y[:2] *= 2.0 ** -1040
    _, yb = _run(H, y)
    # numbers of 2^-1040 hold 34 bits; N rounded products of them
    np.testing.assert_allclose(yb[:2] * 2.0 ** 1000, plain[:2] * 2.0 ** -40, rtol=0,
                               atol=2.0 ** -40 * np.abs(plain[:2]).max() * N * 2.0 ** -32)
    assert np.array_equal(yb[2:], plain[2:])
