"""The epoch-long training kernel, the whole-device gradient pass and the
tree-wise bisection at the sizes where they can go wrong: minibatches smaller
than a pass or than the cluster, one sample over, several passes, a last
minibatch of another size, more epochs than one launch's buffers hold.

Tolerances: an FP32 gradient is within 1e-5 of FP64's largest component, and
a component above 1e-3 of the largest then moves m / sqrt(v) by at most a few
1e-3 of itself at its first steps, i.e. lr * 2e-3 = 2e-6 for lr = 1e-3 (as in
the test of single Adam steps); smaller components are not compared.  Losses:
1e-5 relative at the first epoch, 1e-3 after 48 steps.
"""
import numpy as np
import pytest

from oracle import mlp as M

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def L():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1412_7228_gb300 import lbm
    lbm.lib()
    return lbm


def _data(n, seed):
    rng = np.random.default_rng(seed)
    X = np.stack([rng.uniform(0.6, 0.85, n), rng.uniform(-0.9, -0.8, n), rng.uniform(0, 0.6, n)], 1)
    Y = np.stack([(1 - X[:, 2]) * (0.9 - X[:, 0]) * 0.05, 0.3 + 0.2 * (0.85 - X[:, 0]),
                  0.02 * X[:, 0] ** 3, 1e-3 * (1 + X[:, 1])], 1)
    return X, Y


NORM = (np.array([0.72, -0.85, 0.3]), np.array([0.07, 0.03, 0.17]), np.array([0.006, 0.32, 0.008, 1.5e-4]),
        np.array([0.004, 0.015, 0.002, 3e-5]))


def _mlp(L, n, seed):
    mlp = L.Mlp(max_samples=n, seed=seed)
    mlp.set_normalization(*NORM)
    X, Y = _data(n, seed)
    norm = [v.astype(np.float32).astype(np.float64) for v in NORM]
    Xs = ((X.astype(np.float32) - norm[0]) / norm[1]).astype(np.float32).astype(np.float64)
    Ys = ((Y.astype(np.float32) - norm[2]) / norm[3]).astype(np.float32).astype(np.float64)
    return mlp, X, Y, Xs, Ys


def _reference(p, Xs, Ys, n, epochs, batch, lr, seed):
    """FP64 training with the library's shuffles (Fisher-Yates, splitmix64)."""
    order, state, mask64 = list(range(n)), seed, (1 << 64) - 1
    m, v, t, losses, mask = np.zeros_like(p), np.zeros_like(p), 0, [], np.ones(p.size, dtype=bool)
    for _ in range(epochs):
        for i in range(n - 1, 0, -1):
            state = (state + 0x9E3779B97F4A7C15) & mask64
            z = ((state ^ (state >> 30)) * 0xBF58476D1CE4E5B9) & mask64
            z = ((z ^ (z >> 27)) * 0x94D049BB133111EB) & mask64
            j = (z ^ (z >> 31)) % (i + 1)
            order[i], order[j] = order[j], order[i]
        ls = []
        for f in range(0, n, batch):
            idx = order[f:f + batch]
            l, g = M.loss_grad(p, Xs[idx], Ys[idx])
            mask &= np.abs(g) > 1e-3 * np.abs(g).max()
            t += 1
            p, m, v = M.adam(p, m, v, t, g, lr)
            ls.append(l)
        losses.append(np.mean(ls))
    return p, np.array(losses), mask


@pytest.mark.parametrize("n,batch", [(1, 1), (3, 8), (17, 16), (129, 128), (300, 100), (256, 255), (513, 257),
                                     (1600, 768), (2500, 1024), (6000, 6000)])
def test_one_epoch_matches_fp64(L, n, batch):
    mlp, X, Y, Xs, Ys = _mlp(L, n, n + batch)
    p0 = mlp.get_params().astype(np.float64)
    losses = mlp.train(X, Y, epochs=1, batch=batch, lr=1e-3, seed=5)
    p, want, mask = _reference(p0, Xs, Ys, n, 1, batch, 1e-3, 5)
    assert mask.sum() > 0.5 * mask.size
    assert np.abs(mlp.get_params()[mask] - p[mask]).max() <= 2e-6
    assert abs(losses[0] / want[0] - 1) < 1e-5
    # the same call again from the same start gives the same bits
    q = mlp.get_params()
    mlp.set_params(p0.astype(np.float32))
    again = mlp.train(X, Y, epochs=1, batch=batch, lr=1e-3, seed=5)
    assert np.array_equal(q, mlp.get_params()) and np.array_equal(losses, again)
    mlp.close()


def test_epochs_beyond_one_launch(L):
    """12 epochs of 2000 samples: launches of 1, 2, 4 and 5 epochs over both
    sets of buffers."""
    mlp, X, Y, Xs, Ys = _mlp(L, 2000, 3)
    p0 = mlp.get_params().astype(np.float64)
    losses = mlp.train(X, Y, epochs=12, batch=500, lr=1e-3, seed=7)
    _, want, _ = _reference(p0, Xs, Ys, 2000, 12, 500, 1e-3, 7)
    assert np.abs(losses / want - 1).max() < 1e-3
    mlp.close()


@pytest.mark.parametrize("n", [1, 15, 16, 17, 5000, 12000])
def test_predictions_in_passes(L, n):
    mlp = L.Mlp(max_samples=n, seed=6)
    mlp.set_normalization(*NORM)
    X, _ = _data(n, n)
    norm = [v.astype(np.float32).astype(np.float64) for v in NORM]
    want = M.forward(mlp.get_params().astype(np.float64), (X - norm[0]) / norm[1])[0] * norm[3] + norm[2]
    got = mlp.predict(X)
    assert (np.abs(got - want) <= 1e-5 * np.abs(want).max(0) + 1e-7).all()
    mlp.close()


def test_bisection_is_the_same_in_every_grouping(L):
    """16, 8, 4 or 1 rows of a pass per target (by the number of targets):
    the same midpoints and choices, so the same bits; targets out of range
    give NaN."""
    mlp, X, Y, _, _ = _mlp(L, 2000, 21)
    mlp.train(X, Y, epochs=60, batch=128, lr=3e-3, seed=1)
    rng = np.random.default_rng(9)
    t, A, k = rng.uniform(0.62, 0.83, 41), rng.uniform(-0.88, -0.82, 41), rng.uniform(0.05, 0.55, 41)
    sig = (1 - k) * (0.9 - t) * 0.05
    sig[7], sig[19] = 1.0, -1.0
    first = mlp.invert_kappa(t, A, sig, 0.0, 0.6)
    assert np.isnan(first[[7, 19]]).all() and np.isfinite(np.delete(first, [7, 19])).all()
    for reps in (1, 8, 16, 40):
        got = mlp.invert_kappa(*[np.tile(v, reps) for v in (t, A, sig)], 0.0, 0.6)
        np.testing.assert_array_equal(got.reshape(reps, -1), np.tile(first, (reps, 1)))
    single = np.array([mlp.invert_kappa(t[i:i + 1], A[i:i + 1], sig[i:i + 1], 0.0, 0.6)[0] for i in range(3)])
    np.testing.assert_array_equal(single, first[:3])
    mlp.close()
