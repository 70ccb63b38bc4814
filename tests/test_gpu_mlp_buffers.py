"""Buffers of the network as calls of different kinds and batches follow one another."""
import ctypes

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
f32 = np.float32


def samples(dims, rows):
    rng = np.random.default_rng(rows)
    return rng.normal(0, 1, (rows, dims[0])).astype(f32), rng.normal(0, 1, (rows, dims[-1])).astype(f32)


@pytest.mark.parametrize("path", [0, 1])
@pytest.mark.parametrize("dims", [(7, 2), (109, 6), (20, 32, 3)])
def test_training_after_inference(dims, path):
    from paper_2506_05362_gb300 import pd
    first = pd.MLP(dims, seed=4)
    first.set_forward_path(path)
    X, T = samples(dims, 130)
    want = first.grad(X, T)
    net = pd.MLP(dims, seed=4)
    net.set_forward_path(path)
    net.forward(samples(dims, 200)[0])  # room for 200 rows, none for training
    loss, g = net.grad(X, T)
    assert loss == want[0] and np.array_equal(g, want[1])
    net.forward(samples(dims, 500)[0])  # a larger forward takes the training buffers away
    assert net.train_step(X, T, lr=1e-3) == want[0]
    assert first.train_step(X, T, lr=1e-3) == want[0]
    assert np.array_equal(net.get_params(), first.get_params())
    first.close()
    net.close()


@pytest.mark.parametrize("train", [False, True])
def test_a_refused_allocation_leaves_the_network_usable(train):
    from paper_2506_05362_gb300 import pd
    import torch
    dims = (256, 256)
    X, T = samples(dims, 70)
    net = pd.MLP(dims, seed=5)
    Y, want = net.forward(X), net.grad(X, T)
    Xd, Td = torch.from_numpy(X).cuda(), torch.from_numpy(T).cuda()
    a, b = ctypes.c_void_p(Xd.data_ptr()), ctypes.c_void_p(Td.data_ptr())
    rows = ctypes.c_int64(2 ** 31 - 1)  # a terabyte of activations: refused before anything is launched
    if train:
        status = pd.lib().pd_mlp_train_step_device(net.h, a, b, rows, ctypes.c_float(1e-3), None)
    else:
        status = pd.lib().pd_mlp_forward_device(net.h, a, rows, b)
    assert status == pd.PD_ENOMEM
    assert np.array_equal(net.forward(X), Y)
    loss, g = net.grad(X, T)
    assert loss == want[0] and np.array_equal(g, want[1])
    net.close()
