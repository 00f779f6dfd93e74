"""Every feature of sampled centres against its definition: nearest panels, their
lengths, and the curvature window, in the kernel's staged path and in its path for
boxes with more sources or panels than it stages."""
import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu


def _curvature(g):
    """Turning of the normal between the neighbouring nodes of the panel, one-sided at its ends."""
    nb, n, xy = g["nb"], g["base_n"], g["base_xy"]
    i = np.arange(len(n))
    a, b = np.where(i % nb == 0, i, i - 1), np.where(i % nb == nb - 1, i, i + 1)
    turn = np.arctan2(n[a, 0] * n[b, 1] - n[a, 1] * n[b, 0], (n[a] * n[b]).sum(1))
    return turn / np.hypot(*(xy[b] - xy[a]).T)


@pytest.mark.parametrize("n_max,panels", [(32, 24), (100000, 12), (100000, 140)])
def test_features_of_sampled_centres(n_max, panels):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1801_04070_gb300 import Geometry, params_default
    g = workloads.small_grid(2, 1, panels, 50, seed=5)
    geo = Geometry(g, params_default(p_qbx=4, p_fmm=8, n_max=n_max))
    geo.build()
    f = geo.features()
    L, (so, co, _), (xy, r, _) = geo.lists(), geo.owners(), geo.centres()
    srcs = {b: np.nonzero(so == b)[0] for b in np.unique(so)}
    geo.close()
    nb, nu, kappa = g["nb"], g["nu"], _curvature(g)
    ordered = 0
    for c in np.random.default_rng(0).choice(len(r), 80, replace=False):
        node, b = c // 2, co[c]
        panel = node // nb
        near = np.concatenate([srcs.get(d, np.zeros(0, int)) for n in ("U", "WC", "XC")
                               for d in L[n][1][L[n][0][b]:L[n][0][b + 1]]])
        near = near[near // nu != panel]
        best = np.full(g["npanels"], np.inf)
        np.minimum.at(best, near // nu, np.hypot(*(g["up_xy"][near] - xy[c]).T) / r[c])
        top = np.argsort(best, kind="stable")[:9]
        top = top[np.isfinite(best[top])]
        d, k = best[top], min(8, len(top))
        # FP32 of a quotient rounded twice in FP64
        want = np.concatenate([np.minimum(d[:k], 64.0), np.full(8 - k, 64.0)])
        assert np.abs(f[c, :8] - want).max() <= 64 * 2.0 ** -23
        if (np.diff(d) > 1e-5).all():
            lens = np.concatenate([g["panel_len"][top[:k]] / g["panel_len"][panel], np.zeros(8 - k)])
            assert np.array_equal(f[c, 8:16], lens.astype(np.float32))
            ordered += 1
        win = panel * nb + np.clip(node % nb + np.arange(16) - 8, 0, nb - 1)
        curv = (-1 if c & 1 else 1) * kappa[win] * r[c]
        # FP32 curvature, FP32 radius and their product, and the arctangent's 2^-50
        assert (np.abs(f[c, 16:] - curv) <= 2.0 ** -22 * np.abs(curv) + 1e-12).all()
    assert ordered > 40
