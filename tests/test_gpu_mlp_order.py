"""The order of the predictor's gradient sums, bit for bit: a loop over inputs, units and the samples of a chunk of 64, the
chunks' sums added in order, every product fused (FP32). A sum split over threads or CTAs would round otherwise, and
hundreds of Adam steps carry one such rounding to other weights."""
import numpy as np
import pytest

from paper_2410_14088_gb300 import inputs, qsim

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def fma(a, b, c):
    """a * b + c in FP32 with one rounding: the product is exact in 64 bits, the sum is rounded to odd there, and 53 bits
    are two more than twice 24, so that the second rounding is the only one that shows."""
    p, c = np.float64(a) * np.float64(b), np.float64(c)
    p, c = np.broadcast_arrays(p, c)
    s = p + c
    v = s - p
    err = (p - (s - v)) + (c - v)
    odd = (s.view(np.int64) & 1).astype(bool)
    up = np.nextafter(s, np.where(err > 0, np.inf, -np.inf))
    return np.where((err != 0) & ~odd, up, s).astype(np.float32)


def gradient(p, x, t):
    w1, b1 = p[:64 * 41].reshape(64, 41), p[64 * 41:64 * 41 + 64]
    q = p[64 * 41 + 64:]
    w2, b2, w3, b3 = q[:4096].reshape(64, 64), q[4096:4160], q[4160:4224], q[4224]
    n, zero = len(x), np.float32(0)
    a1 = np.broadcast_to(b1, (n, 64)).copy()
    for j in range(41):
        a1 = fma(w1[:, j], x[:, j:j + 1], a1)
    h1 = np.maximum(a1, zero)
    a2 = np.broadcast_to(b2, (n, 64)).copy()
    for j in range(64):
        a2 = fma(w2[:, j], h1[:, j:j + 1], a2)
    h2 = np.maximum(a2, zero)
    y = np.full(n, b3, np.float32)
    for j in range(64):
        y = fma(w3[j], h2[:, j], y)
    dy = (y - t) * (np.float32(1) / np.float32(n))
    d2 = np.where(h2 > 0, dy[:, None] * w3, zero)
    a = np.zeros((n, 64), np.float32)
    for i in range(64):
        a = fma(d2[:, i:i + 1], w2[i], a)
    d1 = np.where(h1 > 0, a, zero)
    total = np.zeros(qsim.MLP_PARAMS, np.float32)
    for c in range(0, n, 64):
        g = [np.zeros(s, np.float32) for s in ((64, 41), 64, (64, 64), 64, 64, ())]
        for b in range(c, min(c + 64, n)):
            g[0] = fma(d1[b][:, None], x[b], g[0])
            g[1] = g[1] + d1[b]
            g[2] = fma(d2[b][:, None], h1[b], g[2])
            g[3] = g[3] + d2[b]
            g[4] = fma(dy[b], h2[b], g[4])
            g[5] = np.float32(g[5] + dy[b])
        total = total + np.concatenate([np.ravel(v) for v in g])
    return total


@pytest.mark.parametrize("batch", [1, 9, 64, 65, 200])
def test_gradient_sums_in_loop_order(batch):
    u = inputs.uniform_array(17, batch * qsim.TRAIN_ROW).reshape(batch, qsim.TRAIN_ROW).astype(np.float32)
    x, t = np.ascontiguousarray(u[:, :41]), u[:, 41] - np.float32(1.5)
    p = ((inputs.uniform_array(18, qsim.MLP_PARAMS) - 0.5) * 0.5).astype(np.float32)
    _, g = qsim.mlp_loss_grad(torch.from_numpy(p).cuda(), torch.from_numpy(x).cuda(), torch.from_numpy(t).cuda())
    np.testing.assert_array_equal(g.cpu().numpy(), gradient(p, x, t))
