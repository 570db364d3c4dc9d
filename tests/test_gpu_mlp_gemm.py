"""Products of the control-variate network at the edges of their tiles and K splits, against FP64.

The operands of every product are rounded to BF16 (unit roundoff u = 2^-8) and summed in FP32.  With
hidden layers scaled so that |pre-activation| stays O(1), a tensor passes at most 7 products (four
forward, three back), each of which perturbs both operands by u at most, and tanh and tanh' pass an error on with a
factor of 2 at most.  The rounding errors are independent, so a tensor's error in the 2-norm stays
below 2 u sqrt(2 * 7) = 0.03 of it; one missing row, column or K step of 64 at these sizes leaves a
larger one in the elements that it reaches, which are compared one by one at 8 u of their tensor's largest."""
import numpy as np
import pytest

from oracle import mlp as omlp
from paper_2601_21005_gb300 import build

import gpu_common as gc

torch = pytest.importorskip('torch')
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize('n_in,width,n_out,rows', [
    (3, 5, 7, 4),                   # less than one copy of 16 bytes
    (20, 64, 40, 5),
    (65, 63, 129, 33),              # one more or less than a tile
    (148, 256, 1603, 32),           # K split over a cluster of 8
    (64, 200, 900, 31),             # a cluster of 4
    (8, 136, 400, 129),             # a cluster of 2
    (37, 1600, 1000, 70),           # hidden layers split too
    (148, 256, 1603, 600),          # 64-row tiles forward
])
def test_products_at_tile_and_split_edges(n_in, width, n_out, rows):
    assert torch.cuda.is_available()
    build.build()
    from paper_2601_21005_gb300 import sgw
    rng = np.random.default_rng(n_in + width + n_out + rows)
    p = omlp.init_params(n_in, width, n_out, seed=5)
    for i in range(1, 8, 2):
        p[i] = 0.1 * rng.normal(size=p[i].shape)
    flat = np.concatenate([a.reshape(-1) for a in p]).astype(np.float32)
    q, o = [], 0
    for a in p:
        q.append(flat[o:o + a.size].reshape(a.shape).astype(np.float64))
        o += a.size
    x = rng.normal(size=(rows, n_in)).astype(np.float32)
    t = rng.normal(size=(rows, n_out)).astype(np.float32)
    w = rng.uniform(0.5, 3.0, size=n_out).astype(np.float32)
    net = sgw.MLP(n_in, width, n_out, rows + 3)
    net.set_params(flat)
    net.set_loss_weights(w)
    xd, td = gc.to_dev(x, torch, torch.float32), gc.to_dev(t, torch, torch.float32)
    y = torch.empty(rows, n_out, dtype=torch.float32, device='cuda')
    loss, g = net.gradients(xd, td, want_grads=True)
    net.forward(xd, y)
    yo, _ = omlp.forward(q, x.astype(np.float64))
    lo, go = omlp.loss_and_grads(q, x.astype(np.float64), t.astype(np.float64), w.astype(np.float64))
    u = 2.0 ** -8
    assert abs(loss - lo) < 0.03 * lo
    got, o = [y.cpu().numpy()], 0
    for a in go:
        got.append(g[o:o + a.size].reshape(a.shape))
        o += a.size
    for k, (a, b) in enumerate(zip(got, [yo] + go)):
        assert np.linalg.norm(a - b) < 0.03 * np.linalg.norm(b), k
        assert np.abs(a - b).max() < 8 * u * np.abs(b).max(), k
    # the same call again gives the same bits, and a smaller batch after it sees none of its rows
    loss2, g2 = net.gradients(xd, td, want_grads=True)
    assert loss2 == loss and np.array_equal(g, g2)
    if rows > 1:
        m = rows // 2
        _, gs = net.gradients(xd[:m], td[:m], want_grads=True)
        fresh = sgw.MLP(n_in, width, n_out, m)
        fresh.set_params(flat)
        fresh.set_loss_weights(w)
        _, gf = fresh.gradients(xd[:m], td[:m], want_grads=True)
        assert np.array_equal(gs, gf)
