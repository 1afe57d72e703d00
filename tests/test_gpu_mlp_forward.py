"""The one-launch forward pass against the FP64 oracle at its edges: rows around every change of the
rows per CTA, widths of one unit, around a warp and up to the widest, one layer and many.

Tolerance: FP32 sums of at most 512 products through at most six layers, 1e-5 of the largest
output (as in the other forward test); with BF16 weights the oracle gets the rounded weights, the
arithmetic stays FP32."""
import numpy as np
import pytest

from oracle import mlp as M

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("in_dim,hidden,depth,out", [
    (7, 256, 4, 8), (1, 1, 2, 1), (70, 31, 3, 33), (7, 33, 6, 2), (512, 512, 2, 512), (3, 200, 4, 5), (9, 16, 1, 40)])
def test_forward_matches_oracle(in_dim, hidden, depth, out):
    import torch
    from paper_1705_01801_gb300 import lbw
    net = lbw.MLP(in_dim, hidden=hidden, depth=depth, out_dim=out, seed=2)
    rng = np.random.default_rng(5)
    p = (net.get_params() + 0.05 * rng.normal(size=net.nparam)).astype(np.float32)  # biases too
    net.set_params(p)
    dims = M.layer_dims(in_dim, hidden, depth, out)
    Ws, bs = M.unpack(p, dims)
    pb = np.concatenate([np.concatenate([torch.from_numpy(W.astype(np.float32)).bfloat16().float().numpy().ravel(), b])
                         for W, b in zip(Ws, bs)])
    for n in (1, 3, 5, 608, 609, 2433, 9729) if hidden == 256 else (2, 130):
        x = rng.normal(size=(n, in_dim)).astype(np.float32)
        for got, q in ((net.forward(x), p), (net.predict_bf16(x), pb)):
            want = M.forward(q, dims, x)[-1]
            np.testing.assert_allclose(got, want, rtol=0, atol=1e-5 * np.abs(want).max())
    # new parameters reach both copies of the weights
    net.set_params(2 * p)
    want = M.forward(2 * p, dims, x)[-1]
    np.testing.assert_allclose(net.forward(x), want, rtol=0, atol=1e-5 * np.abs(want).max())
    assert np.abs(net.predict_bf16(x) - want).max() <= 0.05 * np.abs(want).max() + 0.05
