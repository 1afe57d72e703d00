"""The forward pass of many rows against the FP64 oracle, at the widths and row counts where its
threads change what they share: units around a warp and up to the widest, outputs so few that the
inputs are split, rows around 2433 (the first of this form), 19,456 (fewer threads per block) and no
multiple of a block's 16.  A row's outputs do not depend on how many come with it.

Tolerance: as for few rows, FP32 sums of at most 512 products, 1e-5 of the largest output."""
import numpy as np
import pytest

from oracle import mlp as M

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("in_dim,hidden,depth,out", [
    (7, 256, 4, 8), (1, 1, 2, 1), (70, 31, 3, 33), (7, 33, 6, 2), (512, 512, 2, 512), (7, 64, 4, 1), (31, 100, 3, 32),
    (40, 300, 2, 65), (9, 16, 1, 40), (300, 8, 3, 400), (512, 12, 2, 9)])
def test_many_rows_match_oracle(in_dim, hidden, depth, out):
    from paper_1705_01801_gb300 import lbw
    net = lbw.MLP(in_dim, hidden=hidden, depth=depth, out_dim=out, seed=2)
    rng = np.random.default_rng(5)
    p = (net.get_params() + 0.05 * rng.normal(size=net.nparam)).astype(np.float32)
    net.set_params(p)
    dims = M.layer_dims(in_dim, hidden, depth, out)
    x = rng.normal(size=(19473, in_dim)).astype(np.float32)
    want = M.forward(p, dims, x)[-1]
    few = net.forward(x[:600])
    for n in (2433, 2448, 2449, 19455, 19456, 19473):
        got = net.forward(x[:n])
        np.testing.assert_allclose(got, want[:n], rtol=0, atol=1e-5 * np.abs(want).max())
        np.testing.assert_array_equal(got[:600], few)
