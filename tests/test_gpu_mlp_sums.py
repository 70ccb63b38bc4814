"""The sums of a training step over the batch, bit for bit in their stated order: Adam
divides small gradients by their own size, so that sums grouped otherwise lead to other
weights.

One layer with zero weights and biases: the output is zero and the loss gradient is known
on the host.  T is of another size in every split of the batch, so that the FP32 sums over
splits depend on their order, while a split's own sum of products of few bits is exact
whatever the order."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
f32 = np.float32


def tree(s):
    while s.shape[-1] > 1:
        h = s.shape[-1] // 2
        s = s[..., :h] + s[..., h:]
    return s[..., 0]


def bf16(a):
    import torch
    return torch.from_numpy(np.ascontiguousarray(a)).bfloat16().float().numpy()


def bias_sum(z):
    """Columns of z [rows x n]: 1,024 threads take words of 8 rows in turn, two rows at a time."""
    rows, n = z.shape
    r8 = rows // 8
    k = -(-max(r8, 1) // 1024)
    w = np.zeros((n, k * 1024, 4, 2), f32)
    w[:, :r8] = z[:8 * r8].T.reshape(n, r8, 4, 2)
    pairs = (w[..., 0] + w[..., 1]).reshape(n, k, 1024, 4)
    acc = np.zeros((n, 1024), f32)
    for i in range(k):
        for e in range(4):
            acc = acc + pairs[:, i, :, e]
    t = rows - 8 * r8
    acc[:, :t] = acc[:, :t] + z[8 * r8:].T
    return tree(acc)


def loss_sum(d, ldo):
    """Mean square: blocks of 256 elements of the padded rows in FP32, their sums in FP64."""
    rows, nout = d.shape
    sq = np.zeros((rows, ldo), f32)
    sq[:, :nout] = (d.astype(np.float64) ** 2).astype(f32)
    nb = -(-rows * ldo // 256)
    assert nb <= 8192
    part = tree(np.pad(sq.ravel(), (0, 256 * nb - rows * ldo)).reshape(nb, 256)).astype(np.float64)
    part = np.pad(part, (0, -nb % 256)).reshape(-1, 256)
    acc = np.zeros(256)
    for row in part:
        acc = acc + row
    return f32(tree(acc) / (rows * nout))


def split_size(rows, pad_out):
    """Rows of a split: as many splits, at most 128, as give every SM a CTA of a 128-row tile."""
    import torch
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    most = max(1, min(128, sms // -(-pad_out // 128)))
    return 64 * -(-(-(-rows // 64)) // most)


def weight_sum(z, x, size):
    """dW = z^T x: splits of `size` rows, split k into part k mod 8, the parts in turn."""
    parts = np.zeros((8, z.shape[1], x.shape[1]), f32)
    for k in range(-(-len(z) // size)):
        s = slice(k * size, (k + 1) * size)
        p = z[s].astype(np.float64).T @ x[s].astype(np.float64)
        assert np.array_equal(p, p.astype(f32))  # exact in any order
        parts[k % 8] = parts[k % 8] + p.astype(f32)
    t = parts[0]
    for p in parts[1:]:
        t = t + p
    return t


@pytest.mark.parametrize("rows", [1, 63, 129, 4096, 9751, 65536])
@pytest.mark.parametrize("dims", [(40, 6), (200, 16), (256, 130)])
def test_sums_over_the_batch_keep_their_order(dims, rows):
    from paper_2506_05362_gb300 import pd
    if rows * dims[1] > 1 << 20:
        pytest.skip("more than one element of the loss a thread")
    rng = np.random.default_rng(rows + dims[0])
    pad = [-(-d // 16) * 16 for d in dims]
    size = split_size(rows, pad[1])
    X = rng.integers(-3, 4, (rows, dims[0])).astype(f32)
    scale_of = rng.integers(-10, 11, rows // size + 1)[np.arange(rows) // size]
    T = (rng.uniform(1, 2, (rows, dims[1])) * rng.choice([-1.0, 1.0], (rows, dims[1])) *
         np.exp2(scale_of)[:, None]).astype(f32)
    net = pd.MLP(dims)
    net.set_forward_path(2)
    net.set_params(np.zeros(dims[0] * dims[1] + dims[1], f32))
    loss, g = net.grad(X, T)
    net.close()
    z = bf16(-T * (f32(2) / f32(rows * dims[1])))
    g = np.asarray(g)
    assert loss == loss_sum(-T, pad[1])
    assert np.array_equal(g[dims[0] * dims[1]:], bias_sum(z))
    assert np.array_equal(g[:dims[0] * dims[1]].reshape(dims[1], dims[0]), weight_sum(z, X, size))


@pytest.mark.parametrize("rows", [3, 129, 4099])
@pytest.mark.parametrize("dims", [(109, 256, 256, 6), (30, 64, 3), (256, 128, 256, 20)])
def test_the_training_loss_is_that_of_the_inference_output(dims, rows):
    from paper_2506_05362_gb300 import pd
    rng = np.random.default_rng(rows)
    net = pd.MLP(dims, seed=rows)
    net.set_forward_path(2)
    X = rng.normal(0, 2, (rows, dims[0])).astype(f32)
    T = rng.normal(0, 1, (rows, dims[-1])).astype(f32)
    loss, _ = net.grad(X, T)
    assert loss == loss_sum(net.forward(X) - T, -(-dims[-1] // 16) * 16)
    net.close()
