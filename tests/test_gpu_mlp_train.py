"""The size predictor's training on one cluster of CTAs: gradients at the edges of the split of a batch (eight CTAs of
eight samples at a time) against the FP64 oracle, and a whole training run against the same steps made one by one
through the public gradient and Adam calls."""
import numpy as np
import pytest

import oracle
from paper_2410_14088_gb300 import inputs, qsim

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def sample_rows(n, seed):
    u = inputs.uniform_array(seed, n * qsim.TRAIN_ROW).reshape(n, qsim.TRAIN_ROW).astype(np.float32)
    u[:, 41] = -1.5 + u[:, 3] - u[:, 7]
    return u


def start_params(seed):
    """He-uniform weights from splitmix64 and zero biases, and the stream after them (the shuffles' source)."""
    rng, p = inputs.SplitMix64(seed), []
    for out, fan in ((64, 41), (64, 64), (1, 64)):
        u = np.array([rng.uniform() for _ in range(out * fan)])
        p += [((2 * u - 1) * np.sqrt(6.0 / fan)).astype(np.float32), np.zeros(out, np.float32)]
    return np.concatenate(p), rng


@pytest.mark.parametrize("batch", [1, 7, 8, 9, 63, 64, 65, 129, 1000])
def test_gradient_matches_fp64(batch):
    rows, (p, _) = sample_rows(batch, 3), start_params(9)
    loss64, g64 = oracle.mlp_loss_grad(p.astype(np.float64), rows[:, :41].astype(np.float64), rows[:, 41].astype(np.float64))
    dev = torch.from_numpy(rows).cuda()
    loss, g = qsim.mlp_loss_grad(torch.from_numpy(p).cuda(), dev[:, :41].contiguous(), dev[:, 41].contiguous())
    # FP32 sums of at most 64 + 64 + 41 products along a path and batch / 64 + 8 partials: below 400 roundings of 2^-24
    assert np.linalg.norm(g.cpu().numpy() - g64) <= 400 * 2.0 ** -24 * np.linalg.norm(g64)
    assert abs(loss - loss64) <= 400 * 2.0 ** -24 * loss64


@pytest.mark.parametrize("rows,batch,epochs", [(1, 1, 3), (64, 64, 3), (65, 64, 2), (37, 100, 3), (100, 16, 2), (130, 65, 2)])
def test_training_is_its_steps(rows, batch, epochs):
    data, (p, rng) = sample_rows(rows, 5), start_params(100)
    dev, p = torch.from_numpy(data).cuda(), torch.from_numpy(p).cuda()
    m, v, t = torch.zeros_like(p), torch.zeros_like(p), 0
    for _ in range(epochs):
        order = list(range(rows))
        for i in range(rows - 1, 0, -1):
            j = rng.next_u64() % (i + 1)
            order[i], order[j] = order[j], order[i]
        for b in range(0, rows, batch):
            part = dev[order[b:b + batch]]
            _, g = qsim.mlp_loss_grad(p, part[:, :41].contiguous(), part[:, 41].contiguous())
            t += 1
            qsim.adam_step(p, g, m, v, t, lr=3e-3)
    loss = qsim.predictor_train(data, epochs=epochs, batch=batch, lr=3e-3, seed=100)
    got = qsim.predictor_get()
    # the same gradient code on the same weights: what may differ is the contraction of Adam's products, a few
    # roundings per step, which 20 steps can carry through the gradients to 1e-5 of the weights at most
    assert np.linalg.norm(got - p.cpu().numpy()) <= 1e-5 * np.linalg.norm(got)
    want, _ = qsim.mlp_loss_grad(p, dev[:, :41].contiguous(), dev[:, 41].contiguous())
    assert abs(loss - want) <= 1e-4 * abs(want) + 1e-7
