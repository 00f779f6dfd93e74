"""Direct sums to the QBX centres in fixed point (k_near_centres_fx) against
direct sums in long double: one box holds everything (n_max above the particle
count), so the QBX coefficients are the kernel's alone.

The tolerance is FP64's own for these sums: each term is a product of at most
q + 4 rounded factors and each sum has n terms, (q + 4 + log2 n) 2^-53 of the
absolute sum at worst; the fixed-point terms and sums are rounded below that of
the largest term, which the nearest source's |u| ~ 1 makes part of the sum."""
import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu


def _geo(g, q):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1801_04070_gb300 import Geometry, params_default
    geo = Geometry(g, params_default(p_qbx=q, p_fmm=10, n_max=100000))
    geo.build()
    assert geo.nbox == 1
    return geo


def _problem(panels, nu=64, seed=5):
    g = workloads.starfish.discretize([workloads.Curve(modes=((3, 0.25, 0.3),))], panels, nu=nu)
    rng = np.random.default_rng(seed)
    g["density"] = rng.normal(size=len(g["base_xy"]))
    g["tgt_xy"] = g["base_xy"]
    g["tgt_onsurf"] = np.arange(len(g["base_xy"]), dtype=np.int32)
    return g


def _strengths(g, mu):
    rb, ru = g["ref_b"], g["ref_u"]
    L = np.array([[np.prod([(x - rb[k]) / (rb[j] - rb[k]) for k in range(len(rb)) if k != j]) for j in range(len(rb))]
                  for x in ru])
    return (mu.reshape(-1, len(rb)) @ L.T).ravel() * g["up_w"]


def _reference(g, kern, q, mu, sel, c, r):
    """Coefficients of the centres `sel` and, per order, the absolute sums."""
    f = np.longdouble
    qs = _strengths(g, mu).astype(f)
    st = qs * (g["up_n"][:, 0].astype(f) + 1j * g["up_n"][:, 1].astype(f)) if kern == "D" else qs + 0j
    y = g["up_xy"][:, 0].astype(f) + 1j * g["up_xy"][:, 1].astype(f)
    w = y[None, :] - (c[sel, 0].astype(f) + 1j * c[sel, 1].astype(f))[:, None]
    u = r[sel].astype(f)[:, None] / w
    out, mag = [], []
    for m in range(q + 1):
        if kern == "D":
            t = st / w * u ** m
        elif m == 0:
            t = qs * np.log(np.abs(w)) + 0j
        else:
            t = -st * u ** m / f(m)
        out.append(t.sum(1))
        mag.append(np.abs(t).sum(1))
    return np.stack(out, 1), np.stack(mag, 1)


def _check(g, kern, q, mu=None, sel=None):
    geo = _geo(g, q)
    mu = g["density"] if mu is None else mu
    c, r, _ = geo.centres()
    sel = np.arange(0, len(r), 7) if sel is None else sel
    geo.eval(kern, mu)
    got = geo.qbx_coefficients()[sel] * r[sel, None] ** np.arange(q + 1)
    ref, mag = _reference(g, kern, q, mu, sel, c, r)
    if kern == "S":
        got[:, 0], ref[:, 0] = got[:, 0].real, ref[:, 0].real
    # + 4: the scaling by r^m and its inverse in the export and here
    tol = (q + 8 + np.log2(len(g["up_w"]))) * 2.0 ** -53 * np.maximum(mag, np.abs(_strengths(g, mu)).max())
    assert (np.abs(got - ref) <= tol).all(), (np.abs(got - ref) / tol).max()
    geo.close()


# tiles of 384 sources: below, at and above one and two of them; a warp's 32 lanes not filled
@pytest.mark.parametrize("kern", ["S", "D"])
@pytest.mark.parametrize("panels,nu,q", [(8, 17, 5), (8, 47, 1), (8, 48, 8), (11, 35, 8), (12, 64, 3), (13, 60, 16), (24, 64, 8)])
def test_tile_edges(kern, panels, nu, q):
    _check(_problem(panels, nu), kern, q)


@pytest.mark.parametrize("kern", ["S", "D"])
@pytest.mark.parametrize("dist", [0.97, 0.5, 0.01, 1e-7])
def test_source_inside_the_disk(kern, dist):
    """A source at dist r from a centre: its centre is summed again with the
    distance as radius (1e-7: FP64 order by order for S)."""
    g = _problem(16)
    geo = _geo(g, 8)
    c, r, _ = geo.centres()
    geo.close()
    g["up_xy"] = g["up_xy"].copy()
    g["up_xy"][100] = c[50] + dist * r[50] * np.array([0.6, 0.8])
    _check(g, kern, 8, sel=np.array([50, 51, 200]))


@pytest.mark.parametrize("kern", ["S", "D"])
def test_strength_ranges(kern):
    g = _problem(16)
    mu = g["density"]
    _check(g, kern, 5, mu=np.ldexp(mu, 400))
    _check(g, kern, 5, mu=np.ldexp(mu, -400))
    weak = mu.copy()
    weak[64:] *= 2.0 ** -30
    _check(g, kern, 5, mu=weak)
    geo = _geo(g, 5)
    assert (geo.eval(kern, np.zeros_like(mu)) == 0).all()
    bad = mu.copy()
    bad[3] = np.inf
    assert np.isnan(geo.eval(kern, bad)).all()
    tiny = geo.eval(kern, np.ldexp(mu, -1000))   # outside the scaled range: FP64 sums
    base = geo.eval(kern, mu)
    assert np.abs(np.ldexp(tiny, 1000) - base).max() <= 1e-13 * np.abs(base).max()
    geo.close()


@pytest.mark.parametrize("kern", ["S", "D"])
def test_source_at_a_centre(kern):
    """|w| = 0: NaN for the targets of that centre, the others unharmed."""
    g = _problem(16)
    geo = _geo(g, 5)
    c, r, _ = geo.centres()
    geo.close()
    g["up_xy"] = g["up_xy"].copy()
    g["up_xy"][100] = c[50]
    geo = _geo(g, 5)
    v = geo.eval(kern, g["density"])
    geo.close()
    assert np.isnan(v[25]) and np.isfinite(np.delete(v, 25)).all()
    _check(g, kern, 5, sel=np.array([10, 51, 200]))


@pytest.mark.parametrize("p", [16, 17, 23, 30])
def test_list2_in_fixed_point(p):
    """List 2 of the orders 16 .. 30 (k_m2l_fx) against the FP64 kernels of the
    no-allocation evaluation, on a tree with several levels of List 2 entries
    and odd list lengths.  Both round the far field at 2^-53 of its largest
    terms; 1e-13 is the bound the other List 2 comparisons use."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import ctypes as C

    from paper_1801_04070_gb300 import Geometry, params_default
    from paper_1801_04070_gb300 import _lib
    g = workloads.small_grid(3, 2, 24, 2000, seed=p)
    geo = Geometry(g, params_default(p_qbx=5, p_fmm=p, n_max=32))
    geo.build()
    assert geo.info.list_size[1] > 1000
    dens = torch.tensor(g["density"], dtype=torch.float64, device="cuda")
    for kern in ("S", "D"):
        a = torch.empty(geo.nt, dtype=torch.float64, device="cuda")
        b = torch.empty_like(a)
        geo.eval(kern, dens, a)
        geo._check(geo.L.gq_eval_noalloc(geo._geom, _lib.KERNELS[kern], C.c_void_p(dens.data_ptr()), C.c_void_p(b.data_ptr())))
        torch.cuda.synchronize()
        assert (a - b).abs().max().item() <= 1e-13 * b.abs().max().item(), kern
    geo.close()


@pytest.mark.parametrize("p,q", [(1, 1), (2, 3), (15, 16), (17, 4), (18, 10), (30, 7)])
def test_list3_far_in_fixed_point(p, q):
    """List 3 far at the point targets (k_w_points_fx; odd and even orders) and to
    the centres where the tensor cores do not take it (k_w_centres_fx, p_fmm > 16),
    and the direct sums at the point targets (k_near_points_fx), against the FP64
    kernels of the no-allocation evaluation; the bound as for List 2."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import ctypes as C

    from paper_1801_04070_gb300 import Geometry, params_default
    from paper_1801_04070_gb300 import _lib
    g = workloads.small_grid(2, 2, 20, 4000, seed=p + q)
    geo = Geometry(g, params_default(p_qbx=q, p_fmm=p, n_max=32))
    geo.build()
    assert geo.info.list_size[3] > 1000 and geo.npt > 100
    dens = torch.tensor(g["density"], dtype=torch.float64, device="cuda")
    for kern in ("S", "D"):
        a = torch.empty(geo.nt, dtype=torch.float64, device="cuda")
        b = torch.empty_like(a)
        geo.eval(kern, dens, a)
        geo._check(geo.L.gq_eval_noalloc(geo._geom, _lib.KERNELS[kern], C.c_void_p(dens.data_ptr()), C.c_void_p(b.data_ptr())))
        torch.cuda.synchronize()
        pts = torch.tensor(geo.association()[0] == 0, device="cuda")
        assert (a - b)[pts].abs().max().item() <= 1e-13 * b.abs().max().item(), kern
        # inside-disk sources of these coarse panels amplify the direct sums' rounding by |r/w|^q
        assert (a - b).abs().max().item() <= 1e-13 * b.abs().max().item() * 4.0 ** max(0, q - 5), kern
    geo.close()


@pytest.mark.parametrize("n", [12289, 14335, 14336, 14337])
def test_build_around_the_one_block_sort(n):
    """Particle counts (sources, centres and point targets) far below, just below,
    at and just above the 14,336 of the one-block sort: the same keys have to come
    out in the same stable order, so the tree and owners equal the oracle's."""
    import oracle
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1801_04070_gb300 import Geometry, params_default
    g = workloads.small_grid(1, 1, 128, 20000, seed=2)
    kind, _ = oracle.Oracle(g, oracle.default_params(g)).association()
    base = len(g["up_xy"]) + 2 * len(g["base_xy"])             # 12,288
    points = np.cumsum(kind[:20000] == 0)                      # targets no centre takes
    keep = int(np.searchsorted(points, n - base)) + 1          # the shortest prefix with n - base points
    g["tgt_xy"] = np.ascontiguousarray(g["tgt_xy"][:keep])
    g["tgt_onsurf"] = np.ascontiguousarray(g["tgt_onsurf"][:keep])
    geo = Geometry(g, params_default(p_qbx=5, p_fmm=10, n_max=32))
    geo.build()
    o = oracle.Oracle(g, oracle.default_params(g))
    assert base + o.npt == n
    for a, b in zip(geo.owners(), o.owners()):
        assert np.array_equal(a, b)
    bx, bo = geo.boxes(), o.boxes()
    for k in ("level", "ix", "iy", "parent", "nsrc", "nctr", "ntgt"):
        assert np.array_equal(bx[k], bo[k]), k
    geo.close()


@pytest.mark.parametrize("n", [1, 124, 125, 128, 129, 260, 700])
def test_many_point_targets_in_a_box(n):
    """Point targets of one leaf around the counts at which the four warps of
    k_near_points_fx convert the 32 sums they hold (125 .. 128: the first full
    warp), over two tiles of sources; against long double sums.  The bound is
    64 units of 2^-53 of the terms' absolute sum (logarithm 2 units, products and
    sums below one, conversion and potential's factor 3; 512 terms at random)."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1801_04070_gb300 import Geometry, params_default
    g = workloads.small_grid(1, 1, 8, 0, seed=4)
    rng = np.random.default_rng(n)
    g["tgt_xy"] = np.stack([rng.uniform(-6, 6, n), rng.uniform(3, 6, n)], 1)   # outside every centre's disk
    g["tgt_onsurf"] = np.full(n, -1, np.int32)
    geo = Geometry(g, params_default(p_qbx=5, p_fmm=10, n_max=4000))
    geo.build()
    assert geo.npt == n and geo.info.nbox == 1
    out = np.empty(n)
    geo.eval("S", g["density"], out)
    geo.close()
    q = np.asarray(_strengths(g, g["density"]), np.longdouble)
    d = g["tgt_xy"].astype(np.longdouble)[:, None, :] - g["up_xy"].astype(np.longdouble)[None, :, :]
    terms = q[None, :] * np.log(np.hypot(d[..., 0], d[..., 1]))
    ref = -terms.sum(1) / (2 * np.longdouble(np.pi))
    assert np.all(np.abs(out - ref) <= 64 * 2.0 ** -53 * np.abs(terms).sum(1) / (2 * np.pi))
