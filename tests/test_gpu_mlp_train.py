"""The training step of the surrogate network (two launches per batch) at the
sizes where its tiling changes: one sample, ends of 16- and 64-sample tiles,
and either side of the switch from 16 to 32 samples per CTA (2432), with more
64-sample blocks than the weight-gradient kernel's ring holds (8)."""
import numpy as np
import pytest

from oracle import mlp as ref

pytestmark = pytest.mark.gpu

LO = np.array([0.1, 0.0, 0.2, 0.8])
HI = np.array([1.2, np.pi, 1.6, 2.0])


@pytest.fixture(scope="module")
def wlb():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_2404_02346_gb300 import build as B
    B.build()
    import paper_2404_02346_gb300 as W
    W.lib()
    return W


def _inputs(n, seed):
    rng = np.random.default_rng(seed)
    return LO + (HI - LO) * rng.uniform(size=(n, 4)), rng.standard_normal(n) * 0.5


@pytest.mark.parametrize("n", [1, 15, 17, 64, 65, 513, 2432, 2433])
def test_gradients_match_oracle_at_tile_edges(wlb, n):
    """Per parameter block against FP64 backpropagation with the same BF16
    weights and inputs.  Activations and their gradients are BF16 (relative
    rounding 2^-9 each, eight of them on the longest path): 5 % per block."""
    import torch
    x, t = _inputs(n, n)
    net = wlb.MLP(LO, HI, batch_max=2560)
    net.init_weights(5)
    w = net.get_weights().astype(np.float64)
    loss, g = net.loss_grad(torch.tensor(x, dtype=torch.float32, device="cuda"),
                            torch.tensor(t, dtype=torch.float32, device="cuda"))
    xn = ref.bf16(ref.normalise(x.astype(np.float32).astype(np.float64), LO.astype(np.float32), HI.astype(np.float32)))
    loss_ref, g_ref = ref.loss_and_grad(ref.bf16(w), xn, t.astype(np.float32).astype(np.float64))
    assert loss == pytest.approx(loss_ref, rel=2e-2)
    for name, a, b in zip(["W1", "b1", "W2", "b2", "W3", "b3", "W4", "b4"], ref.unpack(g.astype(np.float64)),
                          ref.unpack(g_ref)):
        assert np.linalg.norm(a - b) <= 5e-2 * np.linalg.norm(b), name
    net.close()


@pytest.mark.parametrize("batch", [128, 640, 2560])
def test_one_training_step_is_adam_on_the_reported_gradient(wlb, batch):
    """One step of train() on a single whole batch moves every weight as Adam
    does with the gradient that loss_grad() reports for those samples (the
    sums over the shuffled samples differ by FP32 rounding, so the bound is a
    hundredth of the step where the gradient is not tiny)."""
    import torch
    x, t = _inputs(batch, 7)
    xt = torch.tensor(x, dtype=torch.float32, device="cuda")
    tt = torch.tensor(t, dtype=torch.float32, device="cuda")
    net = wlb.MLP(LO, HI, batch_max=2560)
    net.init_weights(2)
    w0 = net.get_weights()
    loss, g = net.loss_grad(xt, tt)
    hist = net.train(xt, tt, epochs=1, batch=batch, lr=1e-3, lr_final=1e-3, seed=4)
    step = net.get_weights().astype(np.float64) - w0
    assert hist[0] == pytest.approx(loss, rel=1e-5)
    big = np.abs(g) > 1e-3 * np.abs(g).max()
    # bias-corrected first step: m1 / sqrt(m2) = sign(g)
    assert np.abs(step + 1e-3 * np.sign(g))[big].max() <= 1e-5
    # the packed copies follow the masters: the next gradient sees the new weights
    net2 = wlb.MLP(LO, HI, batch_max=2560)
    net2.set_weights(net.get_weights())
    _, ga = net.loss_grad(xt, tt)
    _, gb = net2.loss_grad(xt, tt)
    assert np.array_equal(ga, gb)
    net.close()
    net2.close()


@pytest.mark.parametrize("n", [1, 16, 17, 2432, 2433, 9728, 9729])
def test_small_predictions_equal_the_layered_forward(wlb, n):
    """Predictions of up to 9728 queries run the forward half of the training
    tiles (16 or 32 queries per CTA), larger ones the persistent kernel: both
    give the bits of the layer-by-layer launches, flags included."""
    import torch
    x, _ = _inputs(n, n)
    x[2::5, 0] = 4.0
    x[3::7, 3] = 0.1
    xt = torch.tensor(x, dtype=torch.float32, device="cuda")
    net = wlb.MLP(LO, HI, batch_max=1024)
    net.init_weights(8)
    y, inside = net.predict(xt)
    net.set_fused(False)
    yl, insl = net.predict(xt)
    assert torch.equal(y, yl) and torch.equal(inside, insl) and torch.isfinite(y).all()
    net.close()
