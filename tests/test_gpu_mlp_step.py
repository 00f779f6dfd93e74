"""The two-launch training step of the order network at batch sizes around its
blocks (8 samples, chunks of 64) against the FP64 network of oracle/mlp.py, and
a training run with awkward columns and batches."""
import numpy as np
import pytest

from oracle import mlp as ref

pytestmark = pytest.mark.gpu


def _net(seed=3):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import workloads
    from paper_1801_04070_gb300 import MLP, Geometry
    geo = Geometry(workloads.unit_circle(8))
    return geo, MLP(geo, seed=seed)


@pytest.mark.parametrize("n", [1, 7, 8, 9, 63, 64, 65, 129, 1000])
def test_gradient_at_block_edges(n):
    geo, m = _net()
    rng = np.random.default_rng(n)
    X = rng.normal(size=(n, 32)).astype(np.float32)
    Y = rng.normal(size=(n, 2)).astype(np.float32)
    loss, grad = m.loss_grad(X, Y)
    l64, g64 = ref.loss_grad(m.weights().astype(np.float64), X.astype(np.float64), Y.astype(np.float64))
    # FP32 sums of n samples: n 2^-24 of the absolute sums at worst, 1e-5 as in the other gradient test
    assert abs(loss - l64) <= 1e-5 * abs(l64)
    assert np.abs(grad - g64).max() <= 1e-5 * np.abs(g64).max()
    m.close()
    geo.close()


def test_standardisation_and_training_reduce_the_error():
    """Columns with a large offset and one constant column (deviation below 1e-6
    counts as 1), a batch that does not divide the set."""
    geo, m = _net()
    rng = np.random.default_rng(0)
    X = (rng.normal(size=(3001, 32)) * rng.uniform(0.1, 30, 32) + rng.normal(size=32) * 50).astype(np.float32)
    X[:, 5] = 2.5
    Y = np.stack([0.3 * X[:, 0] - 0.1 * X[:, 1], np.abs(X[:, 2])], 1).astype(np.float32)
    first = m.train(X, Y, epochs=1, batch=250, lr=1e-3, seed=1)
    last = m.train(X, Y, epochs=20, batch=250, lr=1e-3, seed=1)
    assert np.isfinite(first) and last < 0.3 * first
    p = m.predict(X)
    assert np.isfinite(p).all() and ((p - Y) ** 2).mean() < 0.5 * Y.var()
    m.close()
    geo.close()
