"""GPU: column statistics of closure training, read back exactly, and one Adam
step per parameter.

With a learning rate of 0 and simple weights (W1 the identity on the 16 inputs,
W3 = 1, no biases) the folded weights are the statistics themselves:
W1[k][k] = 1 / sd_k, b1[k] = -mean_k / sd_k, W3 = sd_t, b3 = mean_t.  Mean and
deviation are rounded to FP32 once each and the quotient once: 3 x 2^-24
relative, taken as 4 x 2^-24, plus 1e-9 deviations for the sums of the mean."""
import numpy as np
import pytest

from oracle import closure as ocl

pytestmark = pytest.mark.gpu
ULP = 2.0 ** -24


def cuda(a):
    import torch
    return torch.from_numpy(np.ascontiguousarray(a, dtype=np.float32)).cuda()


def columns(n, rng):
    """Columns of every kind: (values, whether the scale stays 1)."""
    z = rng.standard_normal
    outlier = z(n)
    outlier[0] = 3e4 if n > 1 else 1.0   # the first value far from all others
    late = z(n)
    late[-1] = -3e4 if n > 1 else 1.0
    return [z(n), 1e-25 * z(n), 1e25 * z(n), 1000.0 + 0.01 * z(n), np.full(n, 0.501), outlier, late,
            1e-13 * z(n), 3e18 * z(n), 1e-18 * (1.0 + 0.1 * z(n)), np.zeros(n), 1e-31 * z(n),
            1e37 * (1.0 + 0.1 * z(n)), -5.0 + 1e-3 * z(n), np.where(np.arange(n) == n // 2, 7.0, 0.0),
            np.where(np.arange(n) == 0, 7.0, 0.0)]


@pytest.mark.parametrize("n", [1, 63, 65, 50001, 200000])
@pytest.mark.parametrize("target", [0, 1, 2, 3, 5])
def test_statistics(lbm, n, target):
    rng = np.random.default_rng(n + target)
    X = np.stack(columns(n, rng), axis=1).astype(np.float32)
    t = columns(n, rng)[target].astype(np.float32)
    theta0 = np.zeros(5313)
    theta0[:1024].reshape(64, 16)[np.arange(16), np.arange(16)] = 1.0
    theta0[5248:5312] = 1.0
    theta = cuda(theta0)
    lbm.lbm_closure_train(cuda(X), cuda(t), 1, 1, 0.0, 5, theta)
    th = theta.cpu().numpy().astype(np.float64)
    mu, sd, tm, ts = ocl.standardisation(X, t)
    got = np.diagonal(th[:1024].reshape(64, 16)[:16])
    assert np.all(np.abs(got * sd - 1.0) <= 4 * ULP)
    assert np.all(np.abs(th[1024:1040] + mu / sd) <= 4 * ULP * np.abs(mu / sd) + 1e-9)
    assert np.all(np.abs(th[5248:5312] - ts) <= 4 * ULP * ts)
    assert abs(th[5312] - tm) <= 4 * ULP * abs(tm) + 1e-9 * ts


@pytest.mark.parametrize("n", [65, 50001])
def test_every_parameter_takes_its_step(lbm, n):
    """The first Adam step moves a weight by lr g / (|g| + eps): by lr times the
    gradient's sign wherever |g| stands well above rounding.  In standardised
    coordinates a weight is known to 4 x 2^-24 of itself and, for b1, of the 17
    terms of its folding (each below 2): 2e-5 of the step in all."""
    rng = np.random.default_rng(n)
    X = (rng.standard_normal((n, 16)) * np.logspace(-3, 1, 16) + rng.standard_normal(16) * np.logspace(-3, 1, 16))
    X = X.astype(np.float32)
    t = (0.01 * rng.standard_normal(n) + 0.003).astype(np.float32)
    th0 = np.concatenate([rng.standard_normal(1024) * 0.3, 0.1 * rng.standard_normal(64),
                          rng.standard_normal(4096) * 0.2, 0.1 * rng.standard_normal(64),
                          rng.standard_normal(64) / 8, [0.05]]).astype(np.float32)
    theta, batch, seed, lr = cuda(th0), 96, 5, 0.05
    lbm.lbm_closure_train(cuda(X), cuda(t), 1, batch, lr, seed, theta)
    mu, sd, tm, ts = ocl.standardisation(X, t)
    got = theta.cpu().numpy().astype(np.float64)
    W1 = got[:1024].reshape(64, 16) * sd
    std = np.concatenate([W1.ravel(), got[1024:1088] + W1 @ (mu / sd), got[1088:5248], got[5248:5312] / ts,
                          [(got[5312] - tm) / ts]])
    idx = ocl.minibatch_indices(seed, 1, batch, n)
    _, g = ocl.loss_and_grad(th0.astype(np.float64), (X[idx] - mu) / sd, (t[idx] - tm) / ts)
    step = (th0 - std) / lr
    sizes = {"W1": (0, 1024), "b1": (1024, 1088), "W2": (1088, 5184), "b2": (5184, 5248), "W3": (5248, 5312), "b3": (5312, 5313)}
    for name, (a, b) in sizes.items():
        gb = np.abs(g[a:b])
        clear = gb > 1e-3 * gb.max()
        assert clear.sum() >= (b - a) // 2, name
        want = g[a:b] / (gb + 1e-8)
        assert np.abs(step[a:b] - want)[clear].max() <= 1e-3, name
