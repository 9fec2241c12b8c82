"""The training kernel at the edges of its 128-row tiles: a ragged, a full and a barely started tile, and CTAs that take
several tiles (the accumulators carry over, the last tile is ragged).  Loss and gradients against the oracle, and the
training loop's dependent launches against single steps."""
import numpy as np
import pytest
import torch

from oracle import mlp

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pm():
    from paper_1610_10061_gb300 import pm as mod
    return mod


def _rows(rows, seed):
    rng = np.random.default_rng(seed)
    X = np.zeros((rows, 16))
    X[:, :8] = rng.normal(0, 1, size=(rows, 8))
    X = mlp.bf16_round(X)
    t = rng.normal(0, 1, size=rows)
    return (X, t, torch.from_numpy(X.astype(np.float32)).to(torch.bfloat16).cuda(),
            torch.from_numpy(t.astype(np.float32)).cuda())


def _params(pm, seed):
    params = mlp.init_params(seed=seed)
    for k in ("b1", "b2", "b3"):
        params[k] = np.random.default_rng(seed).normal(0, 0.1, size=params[k].shape)
    return mlp.flatten(params).astype(np.float32)


@pytest.mark.parametrize("rows", [1, 127, 128, 129, -33])
def test_gradients_at_the_edges_of_the_tiles(pm, rows):
    if rows < 0:  # three tiles to a CTA, the last one ragged
        rows = 3 * 128 * torch.cuda.get_device_properties(0).multi_processor_count + rows
    model = pm.Model(seed=1)
    model.set_params(_params(pm, 11))
    p32 = mlp.unflatten(model.params().astype(np.float64))
    X, t, xd, td = _rows(rows, 12)
    loss, g = model.grad(xd, td)
    lref, gref = mlp.loss_and_grads(p32, X, t, bf16=True)
    assert loss == pytest.approx(lref, rel=2e-2)
    G = mlp.unflatten(g.astype(np.float64))
    for name in gref:
        scale = max(1.0, float(np.max(np.abs(gref[name]))))
        np.testing.assert_allclose(G[name], gref[name], rtol=2e-2, atol=1e-3 * scale)


def test_a_training_loop_equals_single_steps(pm):
    """One mini-batch an epoch: the loop's chained launches against the same steps one call each (the sum over the rows
    does not depend on their order but for rounding)."""
    X, t, xd, td = _rows(300, 13)
    start = _params(pm, 14)
    loop, single = pm.Model(seed=1), pm.Model(seed=1)
    loop.set_params(start)
    single.set_params(start)
    losses = loop.train(xd, td, epochs=6, batch=300, lr=1e-3, seed=3)
    ref = [pm.pm_model_train_step(single.handle, xd, td, 300, 1e-3, want_loss=True) for _ in range(6)]
    np.testing.assert_allclose(losses, ref, rtol=1e-3)
