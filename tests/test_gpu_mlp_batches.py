"""The training step's tiles, pieces of the batch and transposed copies at the
edges of their sizes: gradients against the FP64 reference on the features and
weights the kernels use (BF16 operands: 2^-8 a rounding, a handful of them on
each path; the bounds are those of the 1,024-vector check)."""

import numpy as np
import pytest

from oracle import mlp_ref
from paper_2002_09561_gb300 import mdx
from paper_2002_09561_gb300 import workload as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_tx,qam,B", [
    (16, 16, 1), (16, 16, 33), (16, 16, 512), (16, 16, 513), (16, 16, 4160), (16, 16, 8321), (2, 4, 130), (5, 64, 700),
    (32, 64, 129), (32, 16, 640)])
def test_gradients_of_any_batch(n_tx, qam, B):
    import torch

    P = {4: 2, 16: 4, 64: 8}[qam]
    w = wl.generate(9990 + B, B, n_tx, n_tx, qam, 15.0)
    H, y, nv = (torch.from_numpy(w[k]).cuda() for k in ("H", "y", "noise_var"))
    rng = np.random.RandomState(B)
    sym = rng.randint(0, qam, (B, n_tx)).astype(np.uint8)
    met = rng.uniform(0.2, 2.0, B)
    ctx = mdx.Context(0, B, n_tx, n_tx)
    mdx.mlp_init(ctx, n_tx, qam, max_train_batch=B, seed=3)
    params = mdx.make_params(n_tx, n_tx, qam)
    _, feat = mdx.mlp_predict(ctx, params, H, y, nv, want_features=True)
    step = lambda update: mdx.mlp_train_step(ctx, params, H, y, nv, torch.from_numpy(sym).cuda(),  # noqa: E731
                                             torch.from_numpy(met).cuda(), lr=1e-3, update=update, want_grad=True)
    loss, grad = step(False)
    torch.cuda.synchronize()
    d_in, d_out = mdx.mlp_dims(n_tx, qam)
    p = mdx.mlp_get_params(ctx, n_tx, qam).astype(np.float64)
    W1, b1, W2, b2, W3, b3 = mlp_ref.unpack(p, d_in, d_out)
    pr = mlp_ref.pack(mlp_ref.bf16(W1), b1, mlp_ref.bf16(W2), b2, mlp_ref.bf16(W3), b3)
    X = mlp_ref.bf16(feat.cpu().numpy().astype(np.float64))
    lp, lc, ref = mlp_ref.loss_and_grad(pr, X, np.log(met / w["noise_var"]), mlp_ref.targets_to_rows(sym, 2 * n_tx, P),
                                        d_in, d_out, 2 * n_tx, P, round_hidden=mlp_ref.bf16)
    g = grad.cpu().numpy().astype(np.float64)
    assert np.linalg.norm(g - ref) <= 2e-2 * np.linalg.norm(ref)
    assert np.array_equal(g[np.abs(ref) == 0.0], ref[np.abs(ref) == 0.0])  # padding stays zero
    assert loss.cpu().numpy() == pytest.approx([lp, lc], rel=2e-2)
    # the step's own weights are those of the next forward pass
    again = step(True)[1]
    assert torch.equal(grad, again)
    fresh = mdx.Context(0, B, n_tx, n_tx)
    mdx.mlp_init(fresh, n_tx, qam, max_train_batch=B, seed=4)
    mdx.mlp_set_params(fresh, mdx.mlp_get_params(ctx, n_tx, qam))
    assert torch.equal(mdx.mlp_predict(ctx, params, H, y, nv), mdx.mlp_predict(fresh, params, H, y, nv))
    assert mdx.mlp_error(ctx) == 0
