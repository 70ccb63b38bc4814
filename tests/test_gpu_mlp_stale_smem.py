"""Hidden widths that are no multiple of the 64 columns a tensor-core chunk reads: results
do not depend on what an earlier kernel left in shared memory."""
import numpy as np
import pytest

from oracle import mlp as omlp

pytestmark = pytest.mark.gpu
f32 = np.float32


def leave_nans():
    """A full-width network on NaNs: every SM's activation tiles are left full of them."""
    from paper_2506_05362_gb300 import pd
    net = pd.MLP((256, 256, 256, 256), seed=1)
    assert np.isnan(net.forward(np.full((2 * 152 * 128, 256), np.nan, f32))).all()
    net.close()


# inference also takes hidden widths of 16 and 48 columns past a multiple of 64
@pytest.mark.parametrize("dims", [(5, 96, 96, 3), (109, 160, 160, 6), (3, 224, 32, 1), (5, 16, 2), (30, 80, 144, 200, 4)])
@pytest.mark.parametrize("rows", [1, 300, 40000])
def test_results_do_not_depend_on_earlier_kernels(dims, rows):
    from paper_2506_05362_gb300 import pd
    rng = np.random.default_rng(rows + len(dims))
    X = rng.normal(0, 1, (rows, dims[0])).astype(f32)
    T = rng.normal(0, 1, (rows, dims[-1])).astype(f32)
    net = pd.MLP(dims, seed=3)
    net.set_forward_path(2)
    th = net.get_params()
    leave_nans()
    Y = net.forward(X)
    ref = omlp.forward(th.astype(np.float64), X, dims, bf16=True)
    # BF16 storage of input and activations (unit roundoff 2^-9): a flipped rounding moves
    # the output by some 4e-3 of its norm, a gradient by some 3e-2 (four roundings a layer)
    assert np.linalg.norm(Y - ref) <= 4e-3 * np.linalg.norm(ref)
    if all(d % 32 == 0 for d in dims[1:-1]):
        leave_nans()
        loss, g = net.grad(X, T)
        rl, rg = omlp.loss_and_grad(th.astype(np.float64), X, T, dims, bf16=True)
        assert abs(loss - rl) <= 1.2e-2 * rl
        assert np.linalg.norm(g - rg) <= 3e-2 * np.linalg.norm(rg)
        leave_nans()
        assert net.train_step(X, T, lr=1e-3) == loss
        new = net.get_params()
        opt = omlp.Adam(th.astype(np.float64), lr=1e-3)
        opt.step(np.asarray(g, np.float64))
        assert np.allclose(new, opt.theta, rtol=1e-5, atol=1e-7)
    net.close()
