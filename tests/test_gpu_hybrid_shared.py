"""The hybrid where many prefixes stay inside the sphere (a weak last antenna): the CTAs that share a vector's
prefixes, for each number of survivors a lane holds, against the sorting form (a node budget that is never
reached takes every vector there), to the bit."""

import math

import numpy as np
import pytest

from paper_2002_09561_gb300 import mdx
from paper_2002_09561_gb300 import workload as wl

pytestmark = pytest.mark.gpu


def _run(H, y, nv, qam, K, depth, radius, budget=0):
    import torch

    B, N, M = H.shape[:3]
    ctx = mdx.Context(0, B, N, M)
    args = [torch.from_numpy(x).cuda() for x in (H, y, nv)]
    out = mdx.detect_hybrid(ctx, mdx.make_params(N, M, qam, radius=radius, K=K, depth=depth, budget=budget), *args,
                            want_stats=False)
    return [t.cpu().numpy() for t in out[:3]]


def _weak_last_antenna(M, qam, B, snr, weak, seed):
    w = wl.generate(seed, B, M, M, qam, snr)
    H, p, a = w["H"].copy(), math.isqrt(qam), math.sqrt(1.5 / (qam - 1))
    H[:, :, -1] *= weak
    s = ((2 * (w["sym"] // p) - (p - 1)) + 1j * (2 * (w["sym"] % p) - (p - 1))) * a
    r = np.einsum("bnm,bm->bn", H[..., 0] + 1j * H[..., 1], s)
    noise = np.random.default_rng(seed).standard_normal((B, M, 2)) * np.sqrt(w["noise_var"] / 2)[:, None, None]
    return H, np.stack([r.real, r.imag], 2) + noise, w["noise_var"]


def _prefixes_inside(H, y, qam, depth, metric):
    """How many prefixes are nearer than the metric (FP64, by numpy's QR)."""
    p = math.isqrt(qam)
    lev = (2 * np.arange(p) - (p - 1)) * math.sqrt(1.5 / (qam - 1))
    Q, R = np.linalg.qr(H[..., 0] + 1j * H[..., 1])
    ph = np.diag(R) / np.abs(np.diag(R))
    R, yb = R / ph[:, None], (Q * ph).conj().T @ (y[..., 0] + 1j * y[..., 1])
    n = 2 * R.shape[0]
    T = np.kron(R.real, np.eye(2)) + np.kron(R.imag, np.array([[0.0, -1.0], [1.0, 0.0]]))
    z = np.stack([yb.real, yb.imag], 1).ravel()
    d, x = np.zeros(1), np.zeros((1, 0))
    for i in range(n - 1, n - 1 - depth, -1):
        c = z[i] - x @ T[i, i + 1:]
        d = (d[:, None] + (c[:, None] - T[i, i] * lev) ** 2).ravel()
        x = np.concatenate([np.tile(lev, len(x))[:, None], np.repeat(x, p, 0)], 1)
    return int((d < metric).sum())


@pytest.mark.parametrize("M,K,depth,B,snr,weak", [
    (16, 33, 3, 200, 22.0, 0.1), (24, 64, 4, 40, 24.0, 0.05), (32, 48, 3, 400, 22.0, 0.1), (100, 64, 4, 5, 26.0, 0.05),
    (24, 32, 4, 40, 24.0, 0.05), (100, 20, 4, 5, 26.0, 0.05), (9, 1, 4, 60, 20.0, 0.05), (48, 64, 3, 30, 22.0, 0.1)])
@pytest.mark.parametrize("radius", ["paper", math.inf])
def test_shared_prefixes_against_the_sorting_form(M, K, depth, B, snr, weak, radius):
    H, y, nv = _weak_last_antenna(M, 64, B, snr, weak, 9950 + M + K)
    sym, met, vst = _run(H, y, nv, 64, K, depth, radius)
    # more than 256 prefixes are left after the first four: the large CTAs'
    left = [_prefixes_inside(H[b], y[b], 64, depth, met[b]) for b in range(min(B, 20))]
    assert np.median(left) > 260, left
    for a, b in zip((sym, met, vst), _run(H, y, nv, 64, K, depth, radius, budget=1 << 62)):
        assert np.array_equal(a, b)
