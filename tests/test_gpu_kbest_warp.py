"""K-best by selection (one vector per warp) at the edges of its forms, and
the vectors it leaves to the sorting kernel (ties at a cut): decisions and
counts against the FP64 oracle."""

import math

import numpy as np
import pytest

import oracle
from paper_2002_09561_gb300 import mdx
from paper_2002_09561_gb300 import workload as wl

pytestmark = pytest.mark.gpu


def _run(w, qam, K, radius=math.inf, flags=0):
    import torch

    B, N, M = w["H"].shape[:3]
    ctx = mdx.Context(0, B, N, M)
    H, y, nv = (torch.from_numpy(w[k]).cuda() for k in ("H", "y", "noise_var"))
    out = mdx.detect_kbest(ctx, mdx.make_params(N, M, qam, radius=radius, K=K, flags=flags), H, y, nv)
    return [t.cpu().numpy() for t in out]


@pytest.mark.parametrize("N,M,qam,K,cplx", [
    (2, 2, 4, 1, False), (3, 3, 16, 31, False), (4, 4, 64, 32, False), (5, 5, 64, 33, False), (9, 9, 16, 64, False),
    (10, 9, 4, 65, False), (8, 8, 64, 128, False), (12, 12, 16, 129, False), (7, 7, 64, 256, False),
    (16, 16, 16, 256, False), (17, 17, 16, 64, False), (33, 32, 64, 16, False),
    (4, 4, 4, 256, True), (5, 5, 16, 32, True), (6, 5, 16, 128, True), (5, 5, 64, 32, True), (4, 4, 64, 33, True)])
def test_selection_forms_against_the_oracle(N, M, qam, K, cplx):
    B = 37
    w = wl.generate(9500 + N + K, B, N, M, qam, 16.0)
    sym, met, vst, st = _run(w, qam, K, flags=mdx.MDX_COMPLEX_TREE if cplx else 0)
    ref = oracle.detect_batch("kbest_complex" if cplx else "kbest", w["H"], w["y"], w["noise_var"], qam, K=K,
                              want_gap=True)
    far = ref["gap"] >= 1e-5  # FP32 may order closer pairs the other way
    assert np.array_equal(sym[far], ref["sym"][far])
    np.testing.assert_allclose(met[far], ref["metric"][far], rtol=1e-5, atol=1e-9)
    assert np.array_equal(st[:, 0], ref["stats"][:, 0]) and (vst == 0).all()


@pytest.mark.parametrize("cplx", [False, True])
def test_ties_at_every_cut(cplx):
    """y = 0 on a diagonal channel: every distance comes several times and ties straddle the cuts; the
    kept children are those of the lower parent rank, then the lower child (exact in FP32 and FP64
    alike), between ordinary vectors."""
    B, M, qam, K = 40, 6, 16, 10
    w = wl.generate(9600, B, M, M, qam, 14.0)
    for b in range(0, B, 3):
        w["H"][b] = 0.0
        for i in range(M):
            w["H"][b, i, i, 0] = 1.0
        w["y"][b] = 0.0
    sym, met, vst, st = _run(w, qam, K, flags=mdx.MDX_COMPLEX_TREE if cplx else 0)
    ref = oracle.detect_batch("kbest_complex" if cplx else "kbest", w["H"], w["y"], w["noise_var"], qam, K=K,
                              want_gap=True)
    tied = np.arange(B) % 3 == 0
    ok = (ref["gap"] >= 1e-5) | tied
    np.testing.assert_allclose(met[ok], ref["metric"][ok], rtol=1e-5, atol=1e-9)
    assert np.array_equal(sym[ok & ~tied], ref["sym"][ok & ~tied])
    assert np.array_equal(st[:, 0], ref["stats"][:, 0]) and (vst == 0).all()


def test_radius_doubling():
    w = wl.generate(9700, 64, 8, 8, 16, 12.0)
    sym, met, vst, st = _run(w, 16, 32, radius=1e-3)
    ref = oracle.detect_batch("kbest", w["H"], w["y"], w["noise_var"], 16, radius=1e-3, K=32, want_gap=True)
    far = ref["gap"] >= 1e-5
    assert np.array_equal(sym[far], ref["sym"][far]) and (vst == mdx.MDX_V_EMPTY_RETRIED).all()
