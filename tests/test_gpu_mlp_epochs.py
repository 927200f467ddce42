"""Every epoch of a training run draws its own order of the samples.  Epoch e of
one call continues the generator that epoch e - 1 left, whose state advances by a
constant per draw, so it must equal a call of one epoch with that seed, bit for
bit: an epoch that trained on a mixture of its order and the next one would not."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

GAMMA, MASK = 0x9E3779B97F4A7C15, (1 << 64) - 1


@pytest.fixture(scope="module")
def wlb():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_2404_02346_gb300 import build as B
    B.build()
    import paper_2404_02346_gb300 as W
    W.lib()
    return W


@pytest.mark.parametrize("n,batch,epochs", [(256, 128, 2), (20000, 512, 5), (300001, 4096, 3)])
def test_epochs_of_one_call_equal_calls_of_one_epoch(wlb, n, batch, epochs):
    import torch
    rng = np.random.default_rng(n)
    lo, hi = np.array([0.1, 0.0, 0.2, 0.8]), np.array([1.2, np.pi, 1.6, 2.0])
    x = torch.tensor(lo + (hi - lo) * rng.uniform(size=(n, 4)), dtype=torch.float32, device="cuda")
    t = torch.tensor(rng.standard_normal(n) * 0.5, dtype=torch.float32, device="cuda")
    seed = 77
    whole = wlb.MLP(lo, hi, batch_max=4096)
    whole.init_weights(3)
    hist = whole.train(x, t, epochs=epochs, batch=batch, lr=1e-3, lr_final=1e-3, seed=seed)
    parts = wlb.MLP(lo, hi, batch_max=4096)
    parts.init_weights(3)
    losses = [parts.train(x, t, epochs=1, batch=batch, lr=1e-3, lr_final=1e-3,
                          seed=(seed + e * (n - 1) * GAMMA) & MASK)[0] for e in range(epochs)]
    assert np.array_equal(hist, np.array(losses, dtype=np.float32))
    assert np.array_equal(whole.get_weights(), parts.get_weights())
    whole.close()
    parts.close()
