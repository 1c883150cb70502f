"""The network's kernels at the edges of their tiles: one to 65 samples, input widths down to 1 and
not a multiple of any load width, against the FP64 oracle (bars of the parity tests: 1e-5 forward,
1e-4 per parameter block)."""
import numpy as np
import pytest

from oracle import nn

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("n_in,batch", [(1, 1), (7, 2), (34, 31), (64, 32), (130, 65), (513, 33), (1058, 14)])
def test_outputs_and_gradient(n_in, batch):
    from paper_2311_05322_gb300 import inversion, mw
    rng = np.random.default_rng(1000 * n_in + batch)
    th = inversion.he_init(n_in, n_in + batch)
    x = rng.normal(size=(batch, n_in)).astype(np.float32)
    t = (rng.normal(size=(batch, 2, 32, 32, 32)) * 0.1).astype(np.float32)
    c = mw.Context(0)
    c.nn_init(n_in, th)
    y = c.nn_infer(x)
    L, g = c.nn_loss_grad(x, t)
    c.close()
    p = nn.unpack(th.astype(np.float64), n_in)
    p["W1"], p["W2"] = nn.bf16_round(p["W1"]), nn.bf16_round(p["W2"])
    yo, _ = nn.forward(p, x.astype(np.float64))
    assert np.linalg.norm(y - yo) <= 1e-5 * np.linalg.norm(yo)
    Lo, go = nn.loss_and_grad(nn.pack(p, n_in), n_in, x.astype(np.float64), t.astype(np.float64))
    assert abs(L - Lo) <= 1e-5 * Lo
    gp, gop = nn.unpack(g.astype(np.float64), n_in), nn.unpack(go, n_in)
    for name, _ in nn.param_shapes(n_in):
        assert np.linalg.norm(gp[name] - gop[name]) <= 1e-4 * np.linalg.norm(gop[name]), name


def test_ragged_training_batches():
    """Epochs whose last batch is short: the losses and parameters of Adam on the oracle's gradients."""
    from paper_2311_05322_gb300 import inversion, mw
    n_in, n, batch = 18, 7, 3
    rng = np.random.default_rng(5)
    th = inversion.he_init(n_in, 3)
    x = rng.normal(size=(n, n_in)).astype(np.float32)
    t = (rng.normal(size=(n, 2, 32, 32, 32)) * 0.1).astype(np.float32)
    c = mw.Context(0)
    c.nn_init(n_in, th)
    # lr * steps = 1e-5 moves the loss by less than the bar: every batch sees the oracle's network
    losses, _ = c.nn_train(x, t, batch=batch, epochs=2, lr=1e-6, seed=9)
    c.close()
    p = nn.unpack(th.astype(np.float64), n_in)
    p["W1"], p["W2"] = nn.bf16_round(p["W1"]), nn.bf16_round(p["W2"])
    Lo, _ = nn.loss_and_grad(nn.pack(p, n_in), n_in, x.astype(np.float64), t.astype(np.float64))
    assert np.all(np.abs(losses - Lo) <= 1e-2 * Lo)
