"""A bounded wait of a tensor-core kernel that gave up (here: its mark, set without one)
leaves the weights alone and is reported once, by the next call that waits."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
f32 = np.float32
DIMS = (20, 64, 32, 3)


def net_and_samples():
    from paper_2506_05362_gb300 import pd
    rng = np.random.default_rng(7)
    return pd.MLP(DIMS, seed=8), rng.normal(0, 1, (150, 20)).astype(f32), rng.normal(0, 1, (150, 3)).astype(f32)


def mark(net):
    from paper_2506_05362_gb300 import pd
    assert pd.lib().pd_mlp_mark_timeout(net.h) == pd.PD_OK


@pytest.mark.parametrize("path", [0, 1])
@pytest.mark.parametrize("call", ["forward", "grad", "train_step", "get_params"])
def test_reported_once_by_the_next_call_that_waits(call, path):
    from paper_2506_05362_gb300 import pd
    net, X, T = net_and_samples()
    net.set_forward_path(path)
    twin, _, _ = net_and_samples()
    twin.set_forward_path(path)
    args = {"forward": (X,), "grad": (X, T), "train_step": (X, T, 1e-3), "get_params": ()}[call]
    net.train_step(X, T, 1e-3)
    twin.train_step(X, T, 1e-3)
    mark(net)
    with pytest.raises(pd.PDError) as e:
        getattr(net, call)(*args)
    assert e.value.status == pd.PD_ETIMEOUT
    assert np.array_equal(net.get_params(), twin.get_params())
    for _ in range(3):  # the step that was not taken does not count in Adam's either
        assert net.train_step(X, T, 1e-3) == twin.train_step(X, T, 1e-3)
    assert np.array_equal(net.get_params(), twin.get_params())
    net.close()
    twin.close()


def test_device_steps_wait_for_the_report():
    from paper_2506_05362_gb300 import pd
    import torch
    net, X, T = net_and_samples()
    twin, _, _ = net_and_samples()
    Xd, Td, loss = torch.from_numpy(X).cuda(), torch.from_numpy(T).cuda(), torch.zeros(1, device="cuda")
    net.train_step_device(Xd, Td, 1e-3, loss)
    twin.train_step(X, T, 1e-3)
    mark(net)
    for _ in range(2):
        net.train_step_device(Xd, Td, 1e-3, loss)
    torch.cuda.synchronize()
    assert np.isnan(loss.item())
    with pytest.raises(pd.PDError):
        net.forward(X)
    assert np.array_equal(net.get_params(), twin.get_params())
    net.train_step_device(Xd, Td, 1e-3, loss)
    assert twin.train_step(X, T, 1e-3) == loss.item()
    assert np.array_equal(net.get_params(), twin.get_params())
    net.close()
    twin.close()
