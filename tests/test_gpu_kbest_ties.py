"""K-best on batches in which children tie at the cuts: that such vectors do not wait for one another (an
identity channel without noise, where every distance is a sum of few squares)."""

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


def _lattice(B, M, qam, seed):
    """Identity channels and noise-free symbols (indices k_re P + k_im)."""
    p = math.isqrt(qam)
    q = np.random.default_rng(seed).integers(0, qam, (B, M))
    H = np.zeros((B, M, M, 2))
    H[:, np.arange(M), np.arange(M), 0] = 1.0
    y = np.stack([2 * (q // p) - (p - 1), 2 * (q % p) - (p - 1)], 2) * math.sqrt(1.5 / (qam - 1))
    return H, y, q


@pytest.mark.parametrize("M,K,B", [(8, 16, 5000), (16, 64, 5000)])
def test_tied_vectors_run_side_by_side(M, K, B):
    """A tied vector runs twice, the second time by the sorting kernel, some three times the first's work;
    eight times an ordinary batch is reached where the vectors wait in a row (20 and more at K = 64)."""
    import torch

    H, y, q = _lattice(B, M, 16, 1)
    w = wl.generate(9800, B, M, M, 16, 14.0)
    nv = torch.from_numpy(w["noise_var"]).cuda()
    ctx, p = mdx.Context(0, B, M, M), mdx.make_params(M, M, 16, K=K)
    tied = [torch.from_numpy(x).cuda() for x in (H, y)]
    plain = [torch.from_numpy(w[k]).cuda() for k in ("H", "y")]
    run = lambda t: mdx.detect_kbest(ctx, p, *t, nv, want_stats=False)  # noqa: E731
    sym, met, vst, _ = run(tied)
    assert np.array_equal(sym.cpu().numpy(), q) and float(met.max()) < 1e-20 and not vst.any()
    assert _time(lambda: run(tied)) < 8 * _time(lambda: run(plain))
