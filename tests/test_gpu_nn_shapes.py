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


@pytest.mark.parametrize("n_in,n,batch", [(18, 7, 3), (33, 5, 4)])
def test_training_follows_adam_on_the_oracle(n_in, n, batch):
    """Several ragged batches per epoch at an ordinary rate: losses and every parameter block against FP64 Adam over
    the same batches, and the BF16 weights that Adam leaves against those of a network made from its parameters.
    Bars: FP32 gradients are within 1e-4 of a block's norm; Adam divides by their size, so the share of entries
    smaller than that (about 1e-4 of them) may step either way, sqrt(4e-4) = 2e-2 of the update's norm, 5e-2 asked;
    the loss moves with gradient times update, where those entries count nothing, 1e-4."""
    from paper_2311_05322_gb300 import inversion, mw
    rng = np.random.default_rng(n_in)
    th0 = inversion.he_init(n_in, 4)
    x = rng.normal(size=(n, n_in)).astype(np.float32)
    t = (rng.normal(size=(n, 2, 32, 32, 32)) * 0.1).astype(np.float32)
    seed, epochs = 9, 3
    c = mw.Context(0)
    c.nn_init(n_in, th0)
    losses, _ = c.nn_train(x, t, batch=batch, epochs=epochs, lr=1e-3, seed=seed)
    th, y = c.nn_get_params(), c.nn_infer(x)
    c.close()
    fresh = mw.Context(0)
    fresh.nn_init(n_in, th)
    assert np.array_equal(y, fresh.nn_infer(x))
    fresh.close()

    ref, mom, var, step, mask = th0.astype(np.float64), 0.0, 0.0, 0, (1 << 64) - 1
    for ep in range(epochs):
        state, perm, total = (seed + 0x632BE59BD9B4E019 * (ep + 1)) & mask, list(range(n)), 0.0
        for i in range(n - 1, 0, -1):       # splitmix64, as the order of an epoch is drawn
            state = z = (state + 0x9E3779B97F4A7C15) & mask
            z = ((z ^ (z >> 30)) * 0xBF58476D1CE4E5B9) & mask
            z = ((z ^ (z >> 27)) * 0x94D049BB133111EB) & mask
            j = (z ^ (z >> 31)) % (i + 1)
            perm[i], perm[j] = perm[j], perm[i]
        for b0 in range(0, n, batch):
            rows = perm[b0:b0 + batch]
            p = nn.unpack(ref, n_in)
            p["W1"], p["W2"] = nn.bf16_round(p["W1"]), nn.bf16_round(p["W2"])
            L, g = nn.loss_and_grad(nn.pack(p, n_in), n_in, x[rows].astype(np.float64), t[rows].astype(np.float64))
            step += 1
            ref, mom, var = nn.adam_step(ref, g, mom, var, step, lr=1e-3)
            total += L * len(rows)
        assert abs(losses[ep] - total / n) <= 1e-4 * total / n, ep
    d, dref = nn.unpack(th.astype(np.float64) - th0, n_in), nn.unpack(ref - th0, n_in)
    for name, _ in nn.param_shapes(n_in):
        assert np.linalg.norm(d[name] - dref[name]) <= 5e-2 * np.linalg.norm(dref[name]), name
