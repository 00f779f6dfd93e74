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


def _features_reference(geo, g):
    """The features straight from their definition, on the host: every source of
    the centre's direct lists measured, panels in order of their nearest source
    (of equal FP32 distances, the one whose source comes first in the lists)."""
    bx, L = geo.boxes(), geo.lists()
    so, co, _ = geo.owners()
    xy, r, _ = geo.centres()
    srcs = [np.nonzero(so == b)[0] for b in range(geo.nbox)]
    nu = g["nu"]
    # sources of a leaf in the library's order: any order gives the same minima
    out = np.zeros((geo.nc, 16), np.float32)
    for c in range(geo.nc):
        b = co[c]
        near = np.concatenate([srcs[d] for n in ("U", "WC", "XC") for d in L[n][1][L[n][0][b]:L[n][0][b + 1]]] + [np.zeros(0, int)])
        near = near[near // nu != c // 2 // g["nb"]]
        dist = (np.hypot(g["up_xy"][near, 0] - xy[c, 0], g["up_xy"][near, 1] - xy[c, 1]) / r[c]).astype(np.float32)
        best = {}
        for p, d in zip((near // nu).tolist(), dist.tolist()):
            best[p] = min(best.get(p, np.inf), d)
        top = sorted(best.items(), key=lambda t: t[1])[:8]
        own = g["panel_len"][c // 2 // g["nb"]]
        out[c, :8] = [min(d, 64.0) for _, d in top] + [64.0] * (8 - len(top))
        out[c, 8:] = [g["panel_len"][p] / own for p, _ in top] + [0.0] * (8 - len(top))
    return out


@pytest.mark.parametrize("n_max,panels", [(32, 24), (2, 12), (4000, 20), (4000, 140)])
def test_nearest_panel_features(n_max, panels):
    """Boxes with few and with many sources (4,000 staged at most; one box holding
    two curves of 140 panels has 17,920 and takes a thread per centre)."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import workloads
    from paper_1801_04070_gb300 import Geometry, params_default
    g = workloads.small_grid(2, 1, panels, 50, seed=5)
    if panels == 140:
        n_max = 100000
    geo = Geometry(g, params_default(p_qbx=4, p_fmm=8, n_max=n_max))
    geo.build()
    f = geo.features()
    ref = _features_reference(geo, g) if panels < 100 else None
    if ref is not None:
        # distances: one rounding of the hypotenuse and one of the division (2 ulp of FP64) before FP32
        assert np.abs(f[:, :8] - ref[:, :8]).max() <= 64 * 2.0 ** -23
        same = np.abs(np.diff(ref[:, :8], axis=1)).min(1) > 1e-5   # no ties: the order is certain
        assert np.array_equal(f[same, 8:16], ref[same, 8:16]) and same.mean() > 0.5
    else:
        assert np.isfinite(f).all() and (np.diff(f[:, :8], axis=1) >= 0).all() and (f[:, 0] > 0).all()
    geo.close()
