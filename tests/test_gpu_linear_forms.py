"""The linear detectors' forms (triangular solve of eight lanes per vector,
MMSE on the augmented QR, normal equations where that QR does not apply) at
the edges of their ranges, against numpy in 64 bits.  A component within
1e-8 half steps of a decision boundary may go either way."""

import numpy as np
import pytest

from paper_2002_09561_gb300 import mdx
from paper_2002_09561_gb300 import workload as wl

pytestmark = pytest.mark.gpu


def _reference(H, y, nv, qam, mmse):
    P = wl.pam_size(qam)
    a = np.sqrt(3.0 / (2.0 * (qam - 1)))
    M = H.shape[2]
    Hc, yc = H[..., 0] + 1j * H[..., 1], y[..., 0] + 1j * y[..., 1]
    x = np.empty((len(Hc), M), complex)
    for b in range(len(Hc)):
        A, r = Hc[b], yc[b]
        if mmse:
            A, r = np.vstack([A, np.sqrt(nv[b]) * np.eye(M)]), np.concatenate([r, np.zeros(M)])
        x[b] = np.linalg.lstsq(A, r, rcond=None)[0]
    u = 0.5 * (np.stack([x.real, x.imag], -1) / a + (P - 1))
    k = np.clip(np.floor(u + 0.5), 0, P - 1)
    edge = (np.abs(u + 0.5 - np.round(u + 0.5)) < 1e-8).any((1, 2))
    s = (2 * k - (P - 1)) * a
    sc = s[..., 0] + 1j * s[..., 1]
    # ||ybar - R s||^2 = ||y - H s||^2 less the part of y outside H's columns
    metric = np.empty(len(Hc))
    for b in range(len(Hc)):
        Q, R = np.linalg.qr(Hc[b])
        metric[b] = np.linalg.norm(Q.conj().T @ yc[b] - R @ sc[b]) ** 2
    return (k[..., 0] * P + k[..., 1]).astype(np.uint8), metric, edge


@pytest.mark.parametrize("mmse", [False, True])
@pytest.mark.parametrize("N,M,qam,B", [
    (1, 1, 4, 5), (2, 2, 16, 1300), (4, 4, 64, 1300), (5, 4, 16, 17), (8, 8, 16, 1217), (9, 9, 4, 1830), (16, 16, 16, 1830),
    (18, 16, 64, 33), (17, 17, 16, 20), (25, 24, 16, 1300), (32, 32, 4, 40)])
def test_linear_forms_at_their_edges(N, M, qam, B, mmse):
    import torch

    w = wl.generate(9400 + N + M + B, B, N, M, qam, 14.0)
    w["noise_var"][0] = 0.0                       # MMSE without noise is zero forcing
    H, y, nv = (torch.from_numpy(w[k]).cuda() for k in ("H", "y", "noise_var"))
    ctx = mdx.Context(0, B, N, M)
    p = mdx.make_params(N, M, qam, flags=mdx.MDX_LINEAR_MMSE if mmse else 0)
    sym, met, vst, st = mdx.detect("linear", ctx, p, H, y, nv)
    ref, metric, edge = _reference(w["H"], w["y"], w["noise_var"], qam, mmse)
    ok = ~edge
    assert ok.mean() > 0.99 and np.array_equal(sym.cpu().numpy()[ok], ref[ok])
    # metrics of the same points: n rounding errors of a few u on ||y||^2 each
    np.testing.assert_allclose(met.cpu().numpy()[ok], metric[ok], rtol=0,
                               atol=64 * M * 2.0 ** -53 * (np.abs(w["y"]) ** 2).sum((1, 2)).max())
    assert (vst == 0).all() and (st[:, 3] == 1).all()


def test_mmse_vectors_left_to_the_normal_equations():
    """A channel entry of 1e-140 scale beside ordinary vectors (out of the fixed-point range), and a
    singular channel (zero column), which is reported."""
    import torch

    B = 1300
    w = wl.generate(9450, B, 8, 8, 16, 14.0)
    w["H"][1] *= 1e-140
    w["H"][2, :, 3] = 0.0
    H, y, nv = (torch.from_numpy(w[k]).cuda() for k in ("H", "y", "noise_var"))
    ctx = mdx.Context(0, B, 8, 8)
    sym, met, vst, _ = mdx.detect("linear", ctx, mdx.make_params(8, 8, 16, flags=mdx.MDX_LINEAR_MMSE), H, y, nv)
    ref, metric, edge = _reference(w["H"], w["y"], w["noise_var"], 16, True)
    keep = ~edge
    keep[1:3] = False
    assert np.array_equal(sym.cpu().numpy()[keep], ref[keep])
    assert vst[2].item() == mdx.MDX_V_SINGULAR and not sym[2].any() and met[2].item() == 0.0
    assert vst[1].item() == mdx.MDX_V_OK and np.isfinite(met[1].item())
