"""Accuracy of the direct sums to the QBX centres where the strengths of one box
are of very different size, against direct sums in long double.

The scale of every tolerance is the centre's own absolute sum, as it is for FP64
arithmetic: each term is a product of at most q + 4 rounded factors and the sum
has n terms, so the error is at most (q + 8 + log2 n) 2^-53 of the absolute sum
(+ 4 in the constant for the scaling by r^m in the export and its inverse here).
Order m counts with the largest absolute sum of the orders up to m (for S without
the logarithms): a term is formed from that of the order before, and a target takes
the sum over the orders; far sources' higher orders are small beside their first."""
import numpy as np
import pytest

from test_gpu_near_fixed import _geo, _problem, _reference

pytestmark = pytest.mark.gpu


def _error(g, kern, q, sel):
    """Largest error of the coefficients of the centres `sel` in units of the
    tolerance."""
    geo = _geo(g, q)
    c, r, _ = geo.centres()
    geo.eval(kern, g["density"])
    got = geo.qbx_coefficients()[sel] * r[sel, None] ** np.arange(q + 1)
    geo.close()
    ref, mag = _reference(g, kern, q, g["density"], sel, c, r)
    if kern == "S":
        got[:, 0], ref[:, 0] = got[:, 0].real, ref[:, 0].real
    first = 1 if kern == "S" else 0
    mag[:, first:] = np.maximum.accumulate(mag[:, first:], axis=1)
    tol = (q + 8 + np.log2(len(g["up_w"]))) * 2.0 ** -53 * mag
    return float((np.abs(got - ref) / tol).max())


def _move_inside(g, q, sources, centre, dist):
    """Moves the sources to distances dist r from a centre, in different directions."""
    geo = _geo(g, q)
    c, r, _ = geo.centres()
    geo.close()
    g["up_xy"] = g["up_xy"].copy()
    a = 0.3 + 2.4 * np.arange(len(sources))
    g["up_xy"][sources] = c[centre] + dist * r[centre] * np.stack([np.cos(a), np.sin(a)], 1)


@pytest.mark.parametrize("kern", ["S", "D"])
@pytest.mark.parametrize("q", [1, 8, 9, 16])
@pytest.mark.parametrize("dist,weight", [(0.9, 0.0), (0.3, 0.0), (0.1, 1e-6), (0.01, 0.0), (1e-3, 1e-12), (1e-7, 0.0)])
def test_weak_source_inside_the_disk(kern, q, dist, weight):
    """A source inside a centre's disk with little strength or none: the sums of
    the others keep their digits."""
    g = _problem(16)
    _move_inside(g, q, [100], 50, dist)
    g["up_w"] = g["up_w"].copy()
    g["up_w"][100] *= weight
    assert _error(g, kern, q, np.array([50, 51, 200])) <= 1


@pytest.mark.parametrize("kern", ["S", "D"])
@pytest.mark.parametrize("count", [2, 33, 400])
def test_many_sources_inside_the_disk(kern, count):
    """Two, more than a warp and more than a tile of sources inside, of strengths
    from nothing to the others' own."""
    g = _problem(16)
    src = 100 + np.arange(count)
    _move_inside(g, 8, src, 50, np.linspace(0.2, 0.95, count)[:, None])
    g["up_w"] = g["up_w"].copy()
    g["up_w"][src] *= np.resize([0.0, 1e-9, 1.0, 1e-3], count)
    assert _error(g, kern, 8, np.array([50, 51, 200])) <= 1
