"""The one-launch training kernel against the FP64 oracle's Adam steps, at the sizes where its
split can go wrong: hidden widths below, at and above a warp's float4s and no multiple of the
neurons per CTA, batches that are no multiple of a warp's rows or too many to keep in shared
memory, one and several outputs, two to five layers, an odd number of steps (the parameters end
in the other buffer) and a continued run (moments carried over).

Every step is compared from the device's own parameters, so nothing accumulates.  Tolerances: FP32
sums over at most 512 terms move outputs by some 1e-6 (the loss to 1e-5) and a gradient entry by
some 1e-7 of the largest; Adam divides by the entry's own size, so the few entries near zero may
move the other way (2 lr): the update agrees to 1e-2 in norm (seven such entries in 140,000)."""
import numpy as np
import pytest

from oracle import mlp as M

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("hidden,out,depth,batch", [
    (256, 8, 4, 64), (256, 1, 4, 32), (256, 3, 4, 50), (200, 5, 3, 17), (64, 9, 5, 16), (96, 2, 2, 128),
    (128, 16, 4, 1), (4, 1, 3, 5), (260, 2, 4, 33), (512, 8, 4, 40), (256, 8, 4, 300)])
def test_training_follows_the_oracle(hidden, out, depth, batch):
    from paper_1705_01801_gb300 import lbw
    rng = np.random.default_rng(hidden + out)
    n, lr, steps = 320, 1e-3, (5, 7)
    x = rng.normal(size=(n, 7)).astype(np.float32)
    t = (np.tanh(x @ rng.normal(size=(7, out))) + 0.1 * rng.normal(size=(n, out))).astype(np.float32)
    order = np.concatenate([rng.permutation(n)[:batch] for _ in range(sum(steps))]).astype(np.int32)
    net = lbw.MLP(7, hidden=hidden, depth=depth, out_dim=out, seed=3)
    p = net.get_params().astype(np.float64)
    dims = M.layer_dims(7, hidden, depth, out)
    m1, m2, at = np.zeros_like(p), np.zeros_like(p), 0
    for _ in range(sum(steps)):
        rows = order[at * batch:(at + 1) * batch]
        loss = net.train(x, t, rows, batch, lr)
        lo, g = M.loss_and_grad(p, dims, x[rows].astype(np.float64), t[rows].astype(np.float64))
        assert abs(loss[0] - lo) <= 1e-5 * lo
        po, m1, m2 = M.adam(p, g, m1, m2, at + 1, lr)
        q = net.get_params().astype(np.float64)
        assert np.abs(q - po).max() <= 2.1 * lr
        assert np.linalg.norm(q - po) <= 1e-2 * np.linalg.norm(po - p)
        p, at = q, at + 1
    # the same steps in two calls end where single steps end, bit for bit
    again = lbw.MLP(7, hidden=hidden, depth=depth, out_dim=out, seed=3)
    cut = steps[0] * batch
    again.train(x, t, order[:cut], batch, lr)
    again.train(x, t, order[cut:], batch, lr)
    assert np.array_equal(again.get_params(), net.get_params())
