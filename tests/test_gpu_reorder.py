"""Exact sphere decoding with sorted antennas (calls that ask for no
statistics) against the natural order (calls that do): the same symbols, the
same FP64 metrics bit for bit, and the same per-vector status."""

import math

import numpy as np
import pytest

from paper_2002_09561_gb300 import mdx
from paper_2002_09561_gb300 import workload as wl

pytestmark = pytest.mark.gpu


def _both(ctx, p, H, y, nv):
    import torch

    a = mdx.detect_sd(ctx, p, H, y, nv, want_stats=False)
    b = mdx.detect_sd(ctx, p, H, y, nv, want_stats=True)
    torch.cuda.synchronize()
    for k, name in enumerate(("sym", "metric", "vstatus")):
        assert torch.equal(a[k], b[k]), (name, int((a[k] != b[k]).sum()))
    return b


@pytest.mark.parametrize("N,M,qam,snr,B,radius", [
    (4, 4, 16, 6.0, 33, "paper"), (5, 5, 64, 14.0, 700, math.inf), (9, 8, 16, 6.0, 1300, "paper"),
    (12, 9, 64, 16.0, 500, 0.5), (16, 16, 16, 8.0, 1300, "paper"), (16, 16, 4, 2.0, 1217, math.inf),
    (17, 17, 16, 16.0, 300, "paper"), (24, 24, 16, 18.0, 1900, "paper"), (25, 25, 4, 8.0, 200, 3.0),
    (32, 32, 4, 9.0, 1900, "paper"), (36, 33, 4, 12.0, 40, "paper"),
    (4, 4, 16, 6.0, 511, "paper"), (4, 4, 16, 6.0, 512, "paper"), (8, 8, 16, 8.0, 513, "paper"),
    (9, 9, 16, 8.0, 32, "paper")])
def test_sorted_search_returns_what_the_natural_one_does(N, M, qam, snr, B, radius):
    import torch

    w = wl.generate(9100 + N + M, B, N, M, qam, snr)
    H, y, nv = (torch.from_numpy(w[k]).cuda() for k in ("H", "y", "noise_var"))
    if B > 100:
        H[3, :, 1] = H[3, :, 0]              # singular up to rounding
        H[4, :, M - 1] = 0.0                 # singular
        H[5, :, 2] *= 1e-7                   # nearly so
        y[6] = 0.0
    ctx = mdx.Context(0, B, N, M)
    _both(ctx, mdx.make_params(N, M, qam, radius=radius), H, y, nv)
    if radius == math.inf:
        p = mdx.make_params(N, M, qam, radius=radius)
        a = mdx.detect_sd(ctx, p, H, y, None, want_stats=False)
        b = mdx.detect_sd(ctx, p, H, y, nv, want_stats=True)
        torch.cuda.synchronize()
        assert all(torch.equal(a[k], b[k]) for k in range(3))


def test_status_at_the_edge_of_the_first_sphere():
    """Initial r^2 within FP32 error of the ML distance: the status says whether the natural-order
    search's first sphere was empty, whichever order the search took."""
    import torch

    for i in range(6):
        w = wl.generate(9200 + i, 1, 16, 16, 16, 6.0)
        H, y, nv = (torch.from_numpy(np.repeat(w[k], 64, axis=0)).cuda() for k in ("H", "y", "noise_var"))
        ctx = mdx.Context(0, 64, 16, 16)
        m = mdx.detect_sd(ctx, mdx.make_params(16, 16, 16), H, y, nv)[1][0].item()
        seen = set()
        for d in (0.0, 1e-8, 1e-7, 1e-6, 1e-5, 3e-5, 1e-4, 3e-4, 1e-3, 1e-2):
            for s in (-1.0, 1.0):
                b = _both(ctx, mdx.make_params(16, 16, 16, radius=m * (1.0 + s * d)), H, y, nv)
                seen.update(b[2].tolist())
        assert seen == {mdx.MDX_V_OK, mdx.MDX_V_EMPTY_RETRIED}


def test_sorted_search_with_the_network_and_host_buffers():
    import torch

    from paper_2002_09561_gb300 import train

    B = 3000
    w = wl.generate(9300, B, 16, 16, 16, np.tile([4.0, 8.0, 12.0], B // 3))
    H, y, nv = (torch.from_numpy(w[k]).cuda() for k in ("H", "y", "noise_var"))
    ctx = mdx.Context(0, B, 16, 16)
    train.load_model(ctx, 16, 16)
    p = mdx.make_params(16, 16, 16, radius="paper", flags=mdx.MDX_LEARNED_RADIUS | mdx.MDX_LEARNED_ORDER)
    want = _both(ctx, p, H, y, nv)
    sym, met, vst = np.zeros((B, 16), np.uint8), np.zeros(B), np.zeros(B, np.int32)
    mdx.detect_host("sd", ctx, p, w["H"], w["y"], w["noise_var"], sym, met, vst)
    assert np.array_equal(sym, want[0].cpu().numpy()) and np.array_equal(met, want[1].cpu().numpy())
    assert np.array_equal(vst, want[2].cpu().numpy())


def test_vectors_that_fit_need_no_order():
    """On both sides of the number of places (64 an SM up to 32 rows), with and without an order: the same answers."""
    import torch

    sms = torch.cuda.get_device_properties(0).multi_processor_count
    B = 64 * sms + 1
    w = wl.generate(9477, B, 3, 3, 16, 14.0)
    H, y, nv = (torch.from_numpy(w[k]).cuda() for k in ("H", "y", "noise_var"))
    ctx = mdx.Context(0, B, 3, 3)
    p = mdx.make_params(3, 3, 16, radius="paper")
    every = mdx.detect("sd", ctx, p, H, y, nv)
    most = mdx.detect("sd", ctx, p, H[:-1].contiguous(), y[:-1].contiguous(), nv[:-1].contiguous())
    for a, b in zip(every[:3], most[:3]):
        assert torch.equal(a[:-1], b)
