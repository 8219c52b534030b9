"""The hybrid's forms (one vector per warp, CTAs that share a vector's prefixes,
the sorting form) at the edges of their ranges, against the FP64 oracle."""

import math

import numpy as np
import pytest

import oracle
from paper_2002_09561_gb300 import mdx
from paper_2002_09561_gb300 import workload as wl

pytestmark = pytest.mark.gpu


def _run(w, qam, K, depth, radius, stats=True):
    import torch

    B, N, M = w["H"].shape[:3]
    ctx = mdx.Context(0, B, N, M)
    H, y, nv = (torch.from_numpy(w[k]).cuda() for k in ("H", "y", "noise_var"))
    out = (torch.empty((B, M), dtype=torch.uint8, device="cuda"), torch.empty(B, dtype=torch.float64, device="cuda"),
           torch.empty(B, dtype=torch.int32, device="cuda"),
           torch.empty((B, mdx.STATS), dtype=torch.int64, device="cuda") if stats else None)
    mdx.detect("hybrid", ctx, mdx.make_params(N, M, qam, radius=radius, K=K, depth=depth), H, y, nv, out=out)
    return [t.cpu().numpy() for t in out[:3]]


@pytest.mark.parametrize("N,M,qam,K,depth,snr", [
    (1, 1, 4, 4, 0, 10.0), (1, 1, 64, 1, 2, 20.0), (2, 2, 16, 1, 4, 12.0), (5, 4, 4, 32, 1, 8.0), (4, 4, 16, 33, 3, 14.0),
    (4, 4, 64, 64, 2, 20.0), (4, 4, 64, 65, 2, 20.0), (6, 6, 4, 8, 5, 8.0), (8, 8, 64, 2, 4, 18.0),
    (17, 16, 64, 7, 4, 24.0), (33, 33, 16, 31, 3, 18.0), (64, 64, 4, 64, 4, 12.0), (104, 100, 16, 64, 3, 26.0)])
@pytest.mark.parametrize("radius", ["paper", math.inf, 1e-4])
def test_forms_against_the_oracle(N, M, qam, K, depth, snr, radius):
    """1e-4 leaves the first spheres empty (the noise alone is above it)."""
    B = 29 if M < 100 else 7
    w = wl.generate(9700 + M + K, B, N, M, qam, snr)
    sym, met, vst = _run(w, qam, K, depth, radius, stats=False)
    ref = oracle.detect_batch("hybrid", w["H"], w["y"], w["noise_var"], qam, radius=radius, K=K, depth=depth,
                              want_gap=True)
    far = ref["gap"] >= 1e-5
    assert np.array_equal(sym[far], ref["sym"][far])
    np.testing.assert_allclose(met[far], ref["metric"][far], rtol=1e-5, atol=1e-9)
    assert np.array_equal(vst[far], ref["status"][far])
    # statistics count every pass, which is another route for empty spheres
    for a, b in zip(_run(w, qam, K, depth, radius), (sym, met, vst)):
        assert np.array_equal(a[far], b[far])


def test_ties_everywhere():
    """y = 0 on a diagonal channel: equal distances at every cut, resolved by rank; ordinary vectors between."""
    B, M, qam, K = 24, 6, 16, 10
    w = wl.generate(9800, B, M, M, qam, 16.0)
    for b in range(0, B, 3):
        w["H"][b] = 0.0
        for i in range(M):
            w["H"][b, i, i, 0] = 1.0
        w["y"][b] = 0.0
    sym, met, vst = _run(w, qam, K, 2, math.inf)
    ref = oracle.detect_batch("hybrid", w["H"], w["y"], w["noise_var"], qam, K=K, depth=2, want_gap=True)
    far = (ref["gap"] >= 1e-5) & (np.arange(B) % 3 != 0)
    assert np.array_equal(sym[far], ref["sym"][far])
    # every tied leaf has the same metric
    np.testing.assert_allclose(met, ref["metric"], rtol=1e-5, atol=1e-9)
    assert (vst == 0).all()
