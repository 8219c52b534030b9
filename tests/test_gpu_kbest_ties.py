"""K-best where children tie at the cuts, and where the batch decides between the selecting and the sorting
form: tied vectors do not wait for one another, and the forms agree to the bit."""

import math

import numpy as np
import pytest

from paper_2002_09561_gb300 import mdx
from paper_2002_09561_gb300 import workload as wl

pytestmark = pytest.mark.gpu


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


def _lattice(B, N, M, qam, seed):
    """Identity channels and noise-free symbols (indices k_re P + k_im)."""
    p = math.isqrt(qam)
    q = np.random.default_rng(seed).integers(0, qam, (B, M))
    H = np.zeros((B, N, M, 2))
    H[:, np.arange(M), np.arange(M), 0] = 1.0
    y = np.zeros((B, N, 2))
    y[:, :M] = np.stack([2 * (q // p) - (p - 1), 2 * (q % p) - (p - 1)], 2) * math.sqrt(1.5 / (qam - 1))
    return H, y, q


@pytest.mark.parametrize("M,K,B", [(8, 16, 5000), (16, 64, 5000)])
def test_tied_vectors_run_side_by_side(M, K, B):
    """A tied vector runs twice, the second time by the sorting kernel, some three times the first's work;
    eight times an ordinary batch is reached where the vectors wait in a row (20 and more at K = 64)."""
    import torch

    H, y, q = _lattice(B, M, M, 16, 1)
    w = wl.generate(9800, B, M, M, 16, 14.0)
    nv = torch.from_numpy(w["noise_var"]).cuda()
    ctx, p = mdx.Context(0, B, M, M), mdx.make_params(M, M, 16, K=K)
    tied = [torch.from_numpy(x).cuda() for x in (H, y)]
    plain = [torch.from_numpy(w[k]).cuda() for k in ("H", "y")]
    run = lambda t: mdx.detect_kbest(ctx, p, *t, nv, want_stats=False)  # noqa: E731
    sym, met, vst, _ = run(tied)
    assert np.array_equal(sym.cpu().numpy(), q) and float(met.max()) < 1e-20 and not vst.any()
    assert _time(lambda: run(tied)) < 8 * _time(lambda: run(plain))


@pytest.mark.parametrize("N,M,qam,K,cplx,B", [
    (8, 8, 16, 192, False, 640), (5, 5, 4, 256, False, 640), (16, 16, 4, 129, False, 640), (24, 24, 16, 130, False, 640),
    (33, 33, 4, 4, False, 64), (5, 5, 16, 32, True, 640), (16, 16, 16, 17, True, 640), (6, 6, 64, 16, True, 640),
    (34, 6, 64, 3, True, 2560), (34, 8, 4, 16, True, 2560), (7, 7, 4, 128, True, 640), (12, 12, 16, 128, True, 640),
    (32, 32, 4, 48, True, 640)])
def test_forms_agree_to_the_bit(N, M, qam, K, cplx, B):
    """The same 64 vectors in a small batch (sorted, except K = 4 above 32 rows) and many times over in a
    large one (selected): ordinary ones, lattice points on an identity channel (ties between equally far
    parents: left to the sorting kernel) and received vectors far from the lattice (distances so large that
    unequal ones round to the same FP32 number: ties settled by the parents).  (Above 1,216 matrices the QR
    has another form below 33 receive antennas, with other roundings: 34 of them in the largest batches.)"""
    import torch

    w = wl.generate(9900 + M + K, 64, N, M, qam, 12.0)
    H, y = w["H"].copy(), w["y"].copy()
    H[1::4], y[1::4], _ = _lattice(16, N, M, qam, 2)
    y[2::4] = y[2::4] * 30.0 + 7.0
    flags = mdx.MDX_COMPLEX_TREE if cplx else 0
    outs = []
    for times in (1, B // 64):
        ctx = mdx.Context(0, 64 * times, N, M)
        args = [torch.from_numpy(np.concatenate([x] * times)).cuda() for x in (H, y, w["noise_var"])]
        outs.append(mdx.detect_kbest(ctx, mdx.make_params(N, M, qam, K=K, flags=flags), *args))
    for small, large in zip(*outs):
        assert torch.equal(torch.cat([small] * (B // 64)), large)
