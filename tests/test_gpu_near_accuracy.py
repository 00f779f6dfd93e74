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


def _graded(levels, nu, sides=2):
    """A unit circle whose panels halve in length towards one point, from one side or
    from both: neighbouring panels differ by 2 (at the point by up to 2^levels)."""
    nb = 16
    ref_b, ref_u, w_u = (np.polynomial.legendre.leggauss(n)[k] for n, k in ((nb, 0), (nu, 0), (nu, 1)))
    up = np.pi * 0.5 ** np.arange(levels, -1, -1)
    edges = np.concatenate([-up[::-1] if sides == 2 else np.linspace(-np.pi, 0, 9)[:-1], [0.0], up])
    a, h = edges[:-1, None], np.diff(edges)[:, None] / 2

    def nodes(ref):
        th = (a + h + h * ref).ravel()
        return np.stack([np.cos(th), np.sin(th)], 1)
    w = (h * w_u).ravel()
    b, u = nodes(ref_b), nodes(ref_u)
    n = len(edges) - 1
    density = np.random.default_rng(levels).normal(size=n * nb)
    return dict(npanels=n, nb=nb, nu=nu, ref_b=ref_b, ref_u=ref_u, base_xy=b, base_n=b.copy(), up_xy=u, up_n=u.copy(),
                up_w=w, panel_len=2 * h.ravel(), tgt_xy=b, tgt_onsurf=np.arange(n * nb, dtype=np.int32), density=density)


@pytest.mark.parametrize("kern", ["S", "D"])
@pytest.mark.parametrize("levels,nu,sides", [(8, 16, 2), (16, 16, 2), (22, 16, 2), (22, 64, 2), (12, 24, 1), (20, 24, 1)])
@pytest.mark.parametrize("q", [5, 16])
def test_graded_panels_in_one_box(kern, levels, nu, sides, q):
    g = _graded(levels, nu, sides)
    assert _error(g, kern, q, np.arange(3, 2 * 16 * g["npanels"], 11)) <= 1


def test_densities_with_zeros():
    """Unit densities (one node of one panel) and none at all: tiles without strength."""
    g = _problem(24)
    for i in (0, 77):
        g["density"] = np.zeros(24 * 16)
        g["density"][i] = 1.0
        for kern in ("S", "D"):
            assert _error(g, kern, 8, np.arange(2 * (i // 16) * 16, 2 * (i // 16) * 16 + 32)) <= 1


@pytest.mark.parametrize("kern", ["S", "D"])
@pytest.mark.parametrize("levels", [12, 26])
def test_small_far_boxes(kern, levels):
    """List 3 far with boxes much smaller than their distance: strength only on the
    smallest panels of a graded circle, seen from the large panels' centres (order 30,
    k_w_centres_fx) and from points about 1 away, where log|z| is small (k_w_points_fx).
    Tolerances: the sums of the 30 orders and of the levels round at 2^-53 of the
    absolute sum each (70 in all); for S the potential is A_0 log|z| with |z| rounded at
    2^-53 (and 1.75 with |z|^2 and the logarithm's own rounding)."""
    from paper_1801_04070_gb300 import Geometry, params_default
    from test_gpu_near_fixed import _strengths
    g = _graded(levels, 32)
    rng = np.random.default_rng(levels)
    small = np.repeat(g["panel_len"] < 8 * g["panel_len"].min(), 16)
    g["density"] = np.where(small, 2 + rng.normal(size=len(small)), 0.0)
    a = rng.uniform(0, 2 * np.pi, 400)
    g["tgt_xy"] = np.array([1.0, 0.0]) + rng.uniform(0.95, 1.05, (400, 1)) * np.stack([np.cos(a), np.sin(a)], 1)
    g["tgt_onsurf"] = np.full(400, -1, np.int32)
    q = 7
    geo = Geometry(g, params_default(p_qbx=q, p_fmm=30, n_max=32))
    geo.build()
    out = geo.eval(kern, g["density"])
    pts = np.nonzero(geo.association()[0] == 0)[0]
    assert geo.info.list_size[3] > 100 and len(pts) > 100
    f, s = np.longdouble, _strengths(g, g["density"])
    use = s != 0
    s, n, y = s[use].astype(f), g["up_n"][use].astype(f), g["up_xy"][use].astype(f)
    z = (y[:, 0] + 1j * y[:, 1])[None] - (g["tgt_xy"][pts, 0].astype(f) + 1j * g["tgt_xy"][pts, 1].astype(f))[:, None]
    t = (s * (n[:, 0] + 1j * n[:, 1]) / z).real if kern == "D" else s * np.log(np.abs(z))
    tol = 70 * np.abs(s / z).sum(1) if kern == "D" else 3 * np.abs(s).sum() + 70 * np.abs(t).sum(1)
    assert (np.abs(-2 * np.pi * out[pts] - t.sum(1)) <= tol * 2.0 ** -53).all()
    c, r, _ = geo.centres()
    sel = np.nonzero(np.repeat(np.repeat(g["panel_len"] > 0.05, 16), 2))[0][::7]
    got = geo.qbx_coefficients()[sel] * r[sel, None] ** np.arange(q + 1)
    geo.close()
    ref, mag = _reference(g, kern, q, g["density"], sel, c, r)
    if kern == "S":
        got[:, 0], ref[:, 0] = got[:, 0].real, ref[:, 0].real
        mag[:, 0] += 3 * np.abs(s).sum()
    first = 1 if kern == "S" else 0
    mag[:, first:] = np.maximum.accumulate(mag[:, first:], axis=1)
    assert (np.abs(got - ref) <= 70 * 2.0 ** -53 * mag).all()


@pytest.mark.parametrize("kern", ["S", "D"])
@pytest.mark.parametrize("q", [4, 8, 13])
def test_direct_sums_over_several_boxes(kern, q):
    """A tree of one subdivision: several source ranges a box and no far lists, so that
    the coefficients are the direct sums alone."""
    from paper_1801_04070_gb300 import Geometry, params_default
    g = _problem(16)
    geo = Geometry(g, params_default(p_qbx=q, p_fmm=10, n_max=700))
    geo.build()
    assert geo.nbox > 1 and all(geo.info.list_size[i] == 0 for i in (1, 3, 5))
    c, r, _ = geo.centres()
    sel = np.arange(0, len(r), 5)
    geo.eval(kern, g["density"])
    got = geo.qbx_coefficients()[sel] * r[sel, None] ** np.arange(q + 1)
    geo.close()
    ref, mag = _reference(g, kern, q, g["density"], sel, c, r)
    first = 1 if kern == "S" else 0
    if kern == "S":
        got[:, 0], ref[:, 0] = got[:, 0].real, ref[:, 0].real
    mag[:, first:] = np.maximum.accumulate(mag[:, first:], axis=1)
    tol = (q + 8 + np.log2(len(g["up_w"]))) * 2.0 ** -53 * mag
    assert (np.abs(got - ref) <= tol).all(), (np.abs(got - ref) / tol).max()


@pytest.mark.parametrize("p,q", [(17, 4), (18, 10), (20, 8), (30, 7), (15, 10)])
@pytest.mark.parametrize("kern", ["S", "D"])
def test_far_part_of_high_orders(kern, p, q):
    """List 2, List 3 far and M2M in fixed point against FP64: the no-allocation
    evaluation runs those in FP64 and the direct sums by the same kernel, so that what
    differs are the translations alone, at every p_qbx within the bound of the other
    List 2 and 3 comparisons."""
    import ctypes as C

    import torch
    import workloads
    from paper_1801_04070_gb300 import Geometry, _lib, params_default
    g = workloads.small_grid(2, 2, 20, 4000, seed=p + q)
    geo = Geometry(g, params_default(p_qbx=q, p_fmm=p, n_max=32, m2l=1))
    geo.build()
    assert geo.info.list_size[3] > 1000
    dens = torch.tensor(g["density"], dtype=torch.float64, device="cuda")
    a = torch.empty(geo.nt, dtype=torch.float64, device="cuda")
    b = torch.empty_like(a)
    geo.eval(kern, dens, a)
    geo._check(geo.L.gq_eval_noalloc(geo._geom, _lib.KERNELS[kern], C.c_void_p(dens.data_ptr()), C.c_void_p(b.data_ptr())))
    torch.cuda.synchronize()
    geo.close()
    assert (a - b).abs().max().item() <= 1e-13 * b.abs().max().item()
