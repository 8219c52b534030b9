"""The hybrid where more leaves than it keeps are equally near: one answer, whichever warp or CTA comes first."""

import math

import numpy as np
import pytest

import oracle

from test_gpu_hybrid_shared import _run

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,qam,K,depth", [(6, 16, 1, 4), (6, 16, 2, 4), (5, 16, 1, 5), (4, 64, 1, 4), (8, 4, 1, 4), (8, 4, 3, 4),
                                           (4, 16, 70, 4)])
@pytest.mark.parametrize("unitary", [False, True])
def test_tied_candidates_give_one_answer(M, qam, K, depth, unitary):
    """y = 0 on an identity channel, or on a unitary one: all 2^(2 M) points of the inner corners are equally
    near (on the latter up to rounding, which leaves few different distances), more of them than candidates are
    kept.  Their order of arrival must not show."""
    B = 64
    H = np.zeros((B, M, M, 2))
    H[:, np.arange(M), np.arange(M), 0] = 1.0
    if unitary:
        g = np.random.default_rng(M)
        Q, _ = np.linalg.qr(g.standard_normal((M, M)) + 1j * g.standard_normal((M, M)))
        H[:] = np.stack([Q.real, Q.imag], 2)
    y, nv = np.zeros((B, M, 2)), np.full(B, 0.1)
    ref = oracle.detect_batch("hybrid", H[:1], y[:1], nv[:1], qam, K=K, depth=depth)
    first = None
    for radius in (math.inf, 100.0):
        for _ in range(4):
            sym, met, vst = _run(H, y, nv, qam, K, depth, radius)
            np.testing.assert_allclose(met, ref["metric"][0], rtol=1e-6)
            first = sym[0] if first is None else first
            assert (sym == first).all()
