"""Exact SD without a radius and without noise variances: the largest trees (P^level beyond FP32) are searched
in the sorted antenna order as well.  A call with statistics keeps the natural order, so the time tells: on these
channels the sorted search, its second QR included, takes less than half as long."""

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


def test_open_spheres_of_large_trees_are_sorted():
    import torch

    M, B = 24, 600
    w = wl.generate(77 + M, B, M, M, 64, 30.0)
    H, y = (torch.from_numpy(w[k]).cuda() for k in ("H", "y"))
    ctx, p = mdx.Context(0, B, M, M), mdx.make_params(M, M, 64)
    run = lambda stats: mdx.detect_sd(ctx, p, H, y, None, want_stats=stats)  # noqa: E731
    plain, counted = run(False), run(True)
    assert all(torch.equal(a, b) for a, b in zip(plain[:3], counted[:3]))
    assert _time(lambda: run(False)) < _time(lambda: run(True))
