"""Training on the tcgen05 kernels at the edges of their tiles: one layer, narrow and
full-width layers, batches around 128 rows and the K chunk of 64."""
import numpy as np
import pytest

from oracle import mlp as omlp

pytestmark = pytest.mark.gpu

NETS = [(7, 2), (5, 32, 3), (1, 64, 32, 1), (256, 96, 256, 256), (109, 256, 256, 256, 256, 6)]
# BF16 storage (unit roundoff 2^-9) of the input, each hidden activation and each dZ; the
# output of these nets moves by at most about 4e-3 of its norm where a rounding flips, a
# gradient, whose dZ is rounded at each layer, by about 3e-2 of its norm.  The loss and dY
# see the output's error magnified by |Y| / |Y - T|.
FWD_TOL, GRAD_TOL = 4e-3, 3e-2


@pytest.mark.parametrize("batch", [1, 2, 63, 65, 127, 129, 8191])
@pytest.mark.parametrize("dims", NETS)
def test_gradient_and_adam_at_tile_edges(dims, batch):
    from paper_2506_05362_gb300 import pd
    rng = np.random.default_rng(batch + 1000 * len(dims))
    th = np.concatenate([np.concatenate([rng.uniform(-1.7, 1.7, (o, i)).ravel() / np.sqrt(i),
                                         rng.uniform(-0.1, 0.1, o)]) for i, o in zip(dims, dims[1:])])
    th = th.astype(np.float32)
    X = rng.normal(0, 1, (batch, dims[0])).astype(np.float32)
    T = rng.normal(0, 1, (batch, dims[-1])).astype(np.float32)
    net = pd.MLP(dims)
    net.set_forward_path(2)
    net.set_params(th)
    loss, g = net.grad(X, T)
    rl, rg = omlp.loss_and_grad(th.astype(np.float64), X, T, dims, bf16=True)
    Y = omlp.forward(th.astype(np.float64), X, dims, bf16=True)
    amp = max(1.0, np.linalg.norm(Y) / np.linalg.norm(Y - T))
    assert abs(loss - rl) <= 3 * FWD_TOL * amp * rl
    off = 0
    for i, o in zip(dims, dims[1:]):
        for sl in (slice(off, off + o * i), slice(off + o * i, off + o * i + o)):
            a, r = np.asarray(g[sl], np.float64), rg[sl]
            assert np.linalg.norm(a - r) <= GRAD_TOL * amp * np.linalg.norm(r), (i, o, sl)
        off += o * i + o
    # the fused update: Adam on that gradient, then the new weights in every layout the
    # kernels read, the same as those a fresh net packs
    assert net.train_step(X, T, lr=1e-3) == loss
    opt = omlp.Adam(th.astype(np.float64), lr=1e-3)
    opt.step(g.astype(np.float64))
    new = net.get_params()
    assert np.allclose(new, opt.theta, rtol=1e-5, atol=1e-7)
    fresh = pd.MLP(dims)
    fresh.set_forward_path(2)
    fresh.set_params(new)
    l2, g2 = fresh.grad(X, T)
    l1, g1 = net.grad(X, T)
    assert l1 == l2 and np.array_equal(g1, g2)
    net.close()
    fresh.close()
